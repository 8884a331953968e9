// Convergence check of a Krylov basis on the device, shared by the launches of the general path
// (syk_krylov.cu) and the one-CTA basis of small sectors (syk_small.cu).
#pragma once
#include <cuda_runtime.h>

#include "../../include/syk.h"
#include "syk_cheb.cuh"
#include "syk_tridiag.cuh"

namespace syk {

// What a convergence check leaves for the host, or for the kernels that continue on the device:
// the step all columns accept (0: the basis is not good enough yet), the error bits, the matvec's
// status word, and whether the check left the coefficients of that step in c.
struct CheckRec {
  double sacc;
  int status, apply, have_c, m;  // m: the basis' dimension
};

// Eigendecomposition of T (dimension m) by the calling warp into smd: FULL the whole eigenvector
// matrix Q, else rows 0 and m - 1; d the eigenvalues.  Needs m^2 + 2m + 2 (FULL) or 4m doubles.
template <bool FULL>
__device__ inline bool eig_column(int m, int B, int b, const double* alpha, const double* beta, double* smd, double** d,
                           double** q0, double** qm) {
  const int lane = threadIdx.x & 31;
  double* Q = smd;
  *d = FULL ? Q + m * m : smd;
  double* e = *d + m;
  *q0 = FULL ? Q : e + m;
  *qm = FULL ? Q + (m - 1) * m : *q0 + m;
  for (int k = lane; k < m; k += 32) {
    (*d)[k] = alpha[k * B + b];
    e[k] = k + 1 < m ? beta[k * B + b] : 0.0;
  }
  __syncwarp();
  if constexpr (FULL) {
    return tridiag_eig_warp(m, *d, e, Q, e + m);
  } else {
    bool ok = true;
    if (lane == 0) ok = tridiag_eig_rows(m, *d, e, *q0, *qm);
    ok = __shfl_sync(0xffffffffu, ok, 0);
    __syncwarp();
    return ok;
  }
}

// c[k*B + b] = beta0_b (e^{s z T} e_1)_k from the sums of the expansion (times e^{s z c + w'})
__device__ inline void put_coefs(const cheb::Proj& p, double s, double zr, double zi, double2 y0, double2 y1, double beta0,
                          int B, int b, double2* c) {
  const double wx = s * zr * p.r, wy = s * zi * p.r;
  const double2 f = cexp_scaled(1.0, fma(s * zr, p.c, fabs(wx)), fma(s * zi, p.c, wx < 0.0 ? -wy : wy), 1.0);
  const int k = 2 * (threadIdx.x & 31);
  if (k < p.m) c[k * B + b] = make_double2(beta0 * fma(f.x, y0.x, -f.y * y0.y), beta0 * fma(f.x, y0.y, f.y * y0.x));
  if (k + 1 < p.m)
    c[(k + 1) * B + b] = make_double2(beta0 * fma(f.x, y1.x, -f.y * y1.y), beta0 * fma(f.x, y1.y, f.y * y1.x));
}

// Convergence check of column b by one warp: the estimate at s_target; if it passes, the column
// accepts s_target and its coefficients go to c (*have); else, in the basis' last check, the largest
// step that passes (0 in earlier checks, where only the whole step counts).  Returns the step; error
// bits go to status[0].  smd: the warp's own scratch for `cap` terms of the expansion, 4 (cap + 1)
// doubles (at least 4m); beyond cap, or where the expansion loses digits (cheb::keeps), the
// eigendecomposition.  narrow: relative width of the step search.
constexpr int kCheckDoubles = 4 * (cheb::kMaxTerms + 1);
static_assert(kCheckDoubles >= 4 * SYK_MAX_KRYLOV, "scratch of the eigendecomposition's rows");
static __device__ double check_core(int m, int B, int b, const double* alpha, const double* beta, const double* beta0,
                                    double zr, double zi, double s_target, double tol, bool last, int* status,
                                    double* smd, double2* c, bool* have, int cap = cheb::kMaxTerms,
                                    double narrow = 3e-8) {
  const int lane = threadIdx.x & 31;
  const double bl = beta[(m - 1) * B + b];
  const cheb::Proj p = cheb::load(m, alpha + b, beta + b, B);
  const double2 w = make_double2(s_target * zr * p.r, s_target * zi * p.r);
  const double aw = sqrt(fma(w.x, w.x, w.y * w.y));
  *have = false;
  const int K = cheb::terms(aw), K2 = last ? max(K, cheb::terms(2.0 * fabs(w.x))) : K;
  if (aw <= cheb::kMaxW && K2 <= cap) {
    double2* ck = reinterpret_cast<double2*>(smd);
    double* first = smd + 2 * (cap + 1);
    double* lastv = first + cap + 1;
    cheb::coefs(w, K, ck);
    double2 y0, y1;
    cheb::sum(p, K, K2, ck, y0, y1, last ? first : nullptr, last ? lastv : nullptr);
    const double n2 = cheb::norm2(y0, y1);
    if (cheb::keeps(n2, tol)) {
      if (cheb::estimate(p, bl, y0, y1, n2) <= tol) {
        put_coefs(p, s_target, zr, zi, y0, y1, beta0[b], B, b, c);
        *have = true;
        return s_target;
      }
      return last ? cheb::select(p, bl, s_target, tol, zr, zi, first, lastv, narrow) : 0.0;
    }
    __syncwarp();  // the terms have been read: their memory becomes the decomposition's
  }
  double *d, *q0, *qm;
  const bool ok = eig_column<false>(m, B, b, alpha, beta, smd, &d, &q0, &qm);
  if (!ok && lane == 0) atomicOr(status, 2);
  if (last) return select_step(m, d, q0, qm, bl, s_target, tol, zr, zi);
  return step_error(m, d, q0, qm, bl, s_target, zr, zi) <= tol ? s_target : 0.0;
}

// The coefficients of column b at the step s by one warp (put_coefs), false when they need more than
// `cap` terms or the expansion loses digits (cheb::keeps); smd: 2 (cap + 1) doubles.
static __device__ bool coefs_core(int m, int B, int b, const double* alpha, const double* beta, const double* beta0,
                                  double zr, double zi, double s, double tol, double* smd, double2* c,
                                  int cap = cheb::kMaxTerms) {
  const cheb::Proj p = cheb::load(m, alpha + b, beta + b, B);
  const double2 w = make_double2(s * zr * p.r, s * zi * p.r);
  const double aw = sqrt(fma(w.x, w.x, w.y * w.y));
  const int K = cheb::terms(aw);
  if (aw > cheb::kMaxW || K > cap) return false;
  double2* ck = reinterpret_cast<double2*>(smd);
  cheb::coefs(w, K, ck);
  double2 y0, y1;
  cheb::sum(p, K, K, ck, y0, y1, nullptr, nullptr);
  if (!cheb::keeps(cheb::norm2(y0, y1), tol)) return false;
  put_coefs(p, s, zr, zi, y0, y1, beta0[b], B, b, c);
  return true;
}

}  // namespace syk
