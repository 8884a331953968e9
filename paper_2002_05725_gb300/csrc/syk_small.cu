// One Krylov basis of a small sector in one CTA (Supp. Sec. I.B): normalisation, Lanczos steps and
// convergence checks of a basis as a single launch.
//
// With D x B of a few hundred elements a Lanczos step is 6 to 10 launches of kernels that last a
// few microseconds each and occupy one SM anyway (N = 12, one state, complex128: about 120 us a
// step, of which the row matvec 52 and its epilogue 22).  Here the step runs between barriers of
// one CTA: the matvec from shared memory with the coefficients c_m(x) of every row tabulated
// (they are sums of up to n terms otherwise), Gram-Schmidt and norms by groups of lanes.  All
// arithmetic is FP64 for both vector types; the basis is stored in the vectors' type.  FP64 runs
// at 2 multiply-adds per clock and SM: the launch rule keeps a step's matvec below 2^16 of them,
// about 17 us.  Bound by the latency of the step's dependent FP64 operations and barriers.
// Measured: G(t) at N = 12 on 201 times (401 bases, 3615 matvecs) 375 -> 76 ms (190 us a basis with
// its check, combination and host read); before the check's expansion and the tree reductions it
// took 1188 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <complex>

#include "syk_check.cuh"
#include "syk_cplx.cuh"
#include "syk_krylov.cuh"

namespace syk {
namespace {

constexpr int kThreads = 512;
constexpr int kCheckWarps = 4;  // columns checked at a time
constexpr int kMaxEnds = 64;

struct SmallArgs {
  int D, B, M, m;
  const double2* coef;    // M x D: c_m(x)
  const uint32_t* flips;  // M
  const void* cur;
  void* V;
  double *alpha, *beta, *beta0, *sc;
  int orth, passes;  // kOrthFull: Gram-Schmidt passes
  double bt;
  double zr, zi, s_rem, tol;
  const int* st_apply;
  int* status;
  double2* c;
  CheckRec* rec;
  int nends;
  short ends[kMaxEnds];  // basis dimensions to check at, ascending, the last one m
};

template <typename C>
__device__ __forceinline__ double2 load2(const C* p) {
  const C v = *p;
  return make_double2(v.x, v.y);
}
template <typename C>
__device__ __forceinline__ double2 store2(C* p, double2 v) {  // the value as stored
  C w;
  w.x = v.x;
  w.y = v.y;
  *p = w;
  return make_double2(w.x, w.y);
}

template <typename C>
__global__ void __launch_bounds__(kThreads) k_small_basis(SmallArgs a) {
  extern __shared__ __align__(16) double2 sm2[];
  static_assert(kCheckDoubles % 2 == 0, "the warps' scratch starts on 16-byte boundaries");
  const int n = a.D * a.B, B = a.B, t = threadIdx.x, warp = t >> 5, lane = t & 31;
  double2* u = sm2;                 // current basis vector, unnormalised
  double2* w = u + n;               // H v_j, then the next vector
  double2* hh = w + n;              // projections (m + 1) x B
  // kCheckWarps x check scratch (16-byte aligned: it starts with complex values)
  double* scratch = reinterpret_cast<double*>(hh + (a.m + 1) * B);
  double* sc = scratch + kCheckWarps * kCheckDoubles;  // scales (m + 1) x B
  double* h0 = sc + (a.m + 1) * B;                     // Re h_j summed over the passes, B
  double* sb = h0 + B;                                 // accepted steps, B
  __shared__ int miss;
  C* V = static_cast<C*>(a.V);
  const C* cur = static_cast<const C*>(a.cur);

  // |column b| of w; every warp takes columns
  auto norm2 = [&](int b) {
    double s = 0.0;
    for (int x = lane; x < a.D; x += 32) {
      const double2 v = w[x * B + b];
      s = fma(v.x, v.x, fma(v.y, v.y, s));
    }
    return warp_sum(s);
  };
  for (int e = t; e < n; e += kThreads) w[e] = load2(cur + e);
  __syncthreads();
  for (int b = warp; b < B; b += kThreads / 32) {
    const double nb = sqrt(fmax(norm2(b), 0.0));
    if (lane == 0) {
      if (!isfinite(nb)) atomicOr(a.status, 1);
      a.beta0[b] = nb;
      h0[b] = nb > 0.0 ? 1.0 / nb : 0.0;
      a.sc[b] = sc[b] = 1.0;
    }
  }
  __syncthreads();
  for (int e = t; e < n; e += kThreads) {
    const double f = h0[e % B];
    u[e] = store2(V + e, make_double2(w[e].x * f, w[e].y * f));
  }
  int parts = 1;  // lanes that share a row's masks
  while (parts < 16 && n * parts * 2 <= kThreads) parts *= 2;

  int j = 0;
  for (int q = 0; q < a.nends; ++q) {
    for (; j < a.ends[q]; ++j) {
      __syncthreads();
      // w = sc_j H u_j
      const int per = kThreads / parts, part = t & (parts - 1);
      for (int base = 0; base < n; base += per) {
        const int e = base + t / parts;
        double2 s = make_double2(0.0, 0.0);
        if (e < n) {
          const int x = e / B, b = e - x * B;
          for (int m = part; m < a.M; m += parts) {
            const double2 c = __ldg(&a.coef[m * a.D + x]);
            cmac(s, c.x, c.y, u[(x ^ (int)__ldg(&a.flips[m])) * B + b]);
          }
        }
        for (int o = parts >> 1; o > 0; o >>= 1) {
          s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
          s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        }
        if (e < n && part == 0) {
          const double f = sc[j * B + e % B];
          w[e] = make_double2(s.x * f, s.y * f);
        }
      }
      __syncthreads();
      const int k0 = a.orth == kOrthLocal ? max(0, j - 1) : 0, nk = j + 1 - k0;
      for (int pass = 0; pass < a.passes; ++pass) {
        // hh[k] = sc_k <u_k, w>, eight lanes a dot product (three-term recurrence: k = j only, and
        // beta_{j-1} for the vector before it)
        const int first = a.orth == kOrthLocal ? j : 0, dots = (j + 1 - first) * B;
        for (int base = 0; base < dots; base += kThreads / 8) {
          const int i = base + t / 8;
          double2 s = make_double2(0.0, 0.0);
          if (i < dots) {
            const int k = first + i / B, b = i % B;
            for (int x = t & 7; x < a.D; x += 8) {
              const double2 v = load2(V + (size_t)k * n + x * B + b), y = w[x * B + b];
              s.x = fma(v.x, y.x, fma(v.y, y.y, s.x));
              s.y = fma(v.x, y.y, fma(-v.y, y.x, s.y));
            }
          }
          for (int o = 4; o > 0; o >>= 1) {
            s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
            s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
          }
          if (i < dots && (t & 7) == 0) {
            const int at = first * B + i;
            hh[at] = make_double2(sc[at] * s.x, sc[at] * s.y);
          }
        }
        if (a.orth == kOrthLocal && j > 0)
          for (int b = t; b < B; b += kThreads) hh[(j - 1) * B + b] = make_double2(a.beta[(j - 1) * B + b], 0.0);
        __syncthreads();
        for (int e = t; e < n; e += kThreads) {
          const int b = e % B;
          double2 y = w[e];
          for (int k = k0; k < k0 + nk; ++k) {
            const double2 h = hh[k * B + b];
            const double f = sc[k * B + b];
            cmac(y, -h.x * f, -h.y * f, load2(V + (size_t)k * n + e));
          }
          w[e] = y;
        }
        if (pass == 0)
          for (int b = t; b < B; b += kThreads) h0[b] = 0.0;
        __syncthreads();
        for (int b = t; b < B; b += kThreads) h0[b] += hh[j * B + b].x;
        __syncthreads();
      }
      // the next vector as stored, its norm, the step's scalars
      for (int e = t; e < n; e += kThreads) w[e] = u[e] = store2(V + (size_t)(j + 1) * n + e, w[e]);
      __syncthreads();
      for (int b = warp; b < B; b += kThreads / 32) {
        const double n2 = norm2(b);
        if (lane == 0) {
          const double al = h0[b];
          double be = sqrt(fmax(n2, 0.0));
          if (!isfinite(al) || !isfinite(be)) {
            atomicOr(a.status, 1);
            be = 0.0;
          }
          const double prev = j > 0 ? a.beta[(j - 1) * B + b] : 0.0;
          if (be <= a.bt * (fabs(al) + prev)) be = 0.0;
          a.alpha[j * B + b] = isfinite(al) ? al : 0.0;
          a.beta[j * B + b] = be;
          a.sc[(j + 1) * B + b] = sc[(j + 1) * B + b] = be > 0.0 ? 1.0 / be : 0.0;
        }
      }
    }
    // convergence check of the basis of dimension j
    if (t == 0) miss = 0;
    __syncthreads();
    const bool last = q == a.nends - 1;
    if (warp < kCheckWarps)
      for (int b = warp; b < B; b += kCheckWarps) {
        bool have;
        const double s = check_core(j, B, b, a.alpha, a.beta, a.beta0, a.zr, a.zi, a.s_rem, a.tol, last, a.status,
                                    scratch + warp * kCheckDoubles, a.c, &have);
        if (lane == 0) {
          sb[b] = s;
          if (!have) miss = 1;
        }
        __syncwarp();
      }
    __syncthreads();
    double mn = sb[0];
    for (int b = 1; b < B; ++b) mn = fmin(mn, sb[b]);
    if (last || mn >= a.s_rem) {
      if (t == 0) {
        a.rec->sacc = mn;
        a.rec->status = atomicAdd(a.status, 0);
        a.rec->apply = *a.st_apply;
        a.rec->have_c = !miss;
        a.rec->m = j;
      }
      return;
    }
  }
}

size_t small_smem(int64_t D, int64_t B, int m) {
  return size_t(D) * B * 32 + size_t(m + 1) * B * 24 + size_t(B) * 16 + kCheckWarps * kCheckDoubles * sizeof(double);
}

}  // namespace

bool small_basis_applies(const ApplyParams& P, const KrylovWS& ws) {
  const int64_t masks = P.n4 + P.n2 + 1;
  // 2^14 nonzeros (N = 12 to 16 states, N = 14 to 4, N = 16 one state): four FP64 multiply-adds each
  return ws.B <= 16 && ws.D * ws.B <= 1024 && ws.D * ws.B * masks <= (1 << 14) && !prof_enabled() && ws.m <= kMaxEnds &&
         small_smem(ws.D, ws.B, ws.m) <= 200 * 1024;
}

int launch_small_basis(const ApplyParams& P, int dtype, KrylovWS& ws, int orth, bool two_pass, double bt, const void* cur,
                       std::complex<double> z, double s_rem, double tol, const std::vector<int>& ends, cudaStream_t st) {
  const SmallTables* T = nullptr;
  const int rc = small_tables(P.terms, !P.no_alloc, &T);
  if (rc != SYK_OK) return rc;
  SmallArgs a;
  a.D = int(ws.D);
  a.B = int(ws.B);
  a.M = T->masks;
  a.m = ws.m;
  a.coef = T->coef[P.sector];
  a.flips = T->flips;
  a.cur = cur;
  a.V = ws.V;
  a.alpha = ws.alpha;
  a.beta = ws.beta;
  a.beta0 = ws.beta0;
  a.sc = ws.sc;
  a.orth = orth;
  a.passes = orth == kOrthFull && two_pass ? 2 : 1;
  a.bt = bt;
  a.zr = z.real();
  a.zi = z.imag();
  a.s_rem = s_rem;
  a.tol = tol;
  a.st_apply = P.status;
  a.status = ws.status;
  a.c = ws.c;
  a.rec = reinterpret_cast<CheckRec*>(ws.rec);
  a.nends = int(ends.size());
  for (int i = 0; i < a.nends; ++i) a.ends[i] = short(ends[i]);
  const size_t smem = small_smem(ws.D, ws.B, ws.m);
  if (dtype == SYK_C64) {
    SYK_TRY(ensure_smem_limit((const void*)k_small_basis<float2>, 200 * 1024));
    k_small_basis<float2><<<1, kThreads, smem, st>>>(a);
  } else {
    SYK_TRY(ensure_smem_limit((const void*)k_small_basis<double2>, 200 * 1024));
    k_small_basis<double2><<<1, kThreads, smem, st>>>(a);
  }
  count_launch();
  SYK_CUDA_CHECK(cudaGetLastError());
  return SYK_OK;
}

}  // namespace syk
