// The exponential of the Krylov projection without its eigendecomposition (Supp. Sec. I.B): one
// warp evaluates y = e^{s z T} e_1 for a real symmetric tridiagonal T (m <= 64) by the Chebyshev
// expansion, in FP64.
//
// With the spectrum of T inside [c - r, c + r] (Gershgorin) and w = s z r,
//   e^{s z T} e_1 = e^{s z c} sum_k (2 - delta_k0) I_k(w) t_k,   t_k = T_k((T - c)/r) e_1,
// T_k the Chebyshev polynomials (real vectors: t_{k+1} = 2 (T - c)/r t_k - t_{k-1}) and I_k the
// modified Bessel functions, computed for all k at once by Miller's backward recurrence
// I_{k-1} = I_{k+1} + (2k/w) I_k normalised with e^w = I_0 + 2 sum I_k (Olver et al., NIST
// Handbook, 3.6 and 10.35; Re w < 0 by I_k(-w) = (-1)^k I_k(w)).  About |w| + 10 |w|^{1/3} + 15
// terms reach 1e-17.  Everything stays relative to e^{|Re w|}, which cancels in Saad's estimate;
// the sums' rounding error, about 1e-16 on that scale, does not.  In imaginary time |y| may be far
// below 1 there (Gershgorin's interval is wider than the spectrum, and e_1 has little weight at its
// end), and the error is 1e-16/|y| of y: keeps() says whether that is small enough.
//
// Bound by the latency of dependent FP64 operations (FP64 runs at 1/64 of the FP32 rate here).  The
// implicit QR that gave the same quantities is a chain of about m^2 Givens rotations of them: a
// check took 709 us (N = 32, 16 states, m = 16 to 21) and 957 us (complex128, m = 22), the accepted
// basis another 760 to 880 us; the expansion has 20 to 60 steps of a few operations: 41 to 50 us a
// check, the coefficients of the accepted step included.
#pragma once
#include <cuda_runtime.h>

#include "syk_tridiag.cuh"

namespace syk {
namespace cheb {

// |w| the expansion is used for (beyond it, the eigendecomposition), and its terms; the terms at
// 2 |Re w| give the norm of y.
constexpr double kMaxW = 90.0;
constexpr int kMaxTerms = 256;

__device__ __forceinline__ int terms(double absw) {
  const float x = (float)absw;
  return min(kMaxTerms, (int)ceilf(x + 10.f * cbrtf(x) + 15.f));
}

// Lane l of the warp holds rows 2l and 2l + 1 of 2 (T - c)/r: diagonal a0, a1, off-diagonal bl
// (to row 2l - 1), bm (between the two), br (to row 2l + 2).
struct Proj {
  double a0, a1, bl, bm, br;
  double c, r;
  int m;
};

// alpha, beta: entry k at [k * stride]
__device__ inline Proj load(int m, const double* alpha, const double* beta, int stride) {
  const int l = threadIdx.x & 31, k0 = 2 * l, k1 = k0 + 1;
  Proj p;
  p.m = m;
  const double x0 = k0 < m ? alpha[k0 * stride] : 0.0, x1 = k1 < m ? alpha[k1 * stride] : 0.0;
  p.bl = k0 > 0 && k0 < m ? beta[(k0 - 1) * stride] : 0.0;
  p.bm = k1 < m ? beta[k0 * stride] : 0.0;
  p.br = k1 + 1 < m ? beta[k1 * stride] : 0.0;
  const double g0 = fabs(p.bl) + fabs(p.bm), g1 = fabs(p.bm) + fabs(p.br);
  const double big = 1.7976931348623157e308;
  double lo = big, hi = -big;
  if (k0 < m) {
    lo = x0 - g0;
    hi = x0 + g0;
  }
  if (k1 < m) {
    lo = fmin(lo, x1 - g1);
    hi = fmax(hi, x1 + g1);
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  p.c = 0.5 * (lo + hi);
  p.r = 0.5 * (hi - lo);
  const double f = p.r > 0.0 ? 2.0 / p.r : 0.0;
  p.a0 = k0 < m ? (x0 - p.c) * f : 0.0;
  p.a1 = k1 < m ? (x1 - p.c) * f : 0.0;
  p.bl *= f;
  p.bm *= f;
  p.br *= f;
  return p;
}

// a / b
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
  const double n = 1.0 / fma(b.x, b.x, b.y * b.y);
  return make_double2(fma(a.x, b.x, a.y * b.y) * n, fma(a.y, b.x, -a.x * b.y) * n);
}

// ck[k] = (2 - delta_k0) I_k(w) e^{-w'} for k <= K, w' = +-w with Re w' >= 0, by lane 0.
__device__ inline void coefs(double2 w, int K, double2* ck) {
  if ((threadIdx.x & 31) == 0) {
    const bool neg = w.x < 0.0;
    const double2 v = neg ? make_double2(-w.x, -w.y) : w;
    if (fma(v.x, v.x, v.y * v.y) < 1e-16) {  // I_0 = 1, I_1 = w/2 and nothing else to 1e-17
      const double2 e = make_double2(1.0 - v.x, -v.y);
      ck[0] = e;
      if (K > 0) ck[1] = make_double2(fma(v.x, e.x, -v.y * e.y), fma(v.x, e.y, v.y * e.x));
      for (int k = 2; k <= K; ++k) ck[k] = make_double2(0.0, 0.0);
    } else {
      const double2 iv = cdiv(make_double2(2.0, 0.0), v);
      double2 hi = make_double2(0.0, 0.0), a = make_double2(1e-100, 0.0), sum = make_double2(0.0, 0.0);
      for (int k = K + 4; k >= 0; --k) {  // a = I_k, hi = I_{k+1}
        if (k <= K) ck[k] = a;
        sum.x += a.x;
        sum.y += a.y;
        if (k == 0) break;
        const double ux = k * iv.x, uy = k * iv.y;
        const double2 n = make_double2(fma(ux, a.x, fma(-uy, a.y, hi.x)), fma(ux, a.y, fma(uy, a.x, hi.y)));
        hi = a;
        a = n;
      }
      // sum = I_0 + I_1 + ...; e^w = 2 sum - I_0
      const double2 inv = cdiv(make_double2(2.0, 0.0), make_double2(2.0 * sum.x - a.x, 2.0 * sum.y - a.y));
      for (int k = 0; k <= K; ++k) {
        const double2 q = ck[k];
        const double s = k == 0 ? 0.5 : 1.0;
        ck[k] = make_double2(s * fma(q.x, inv.x, -q.y * inv.y), s * fma(q.x, inv.y, q.y * inv.x));
      }
    }
    if (neg)
      for (int k = 1; k <= K; k += 2) ck[k] = make_double2(-ck[k].x, -ck[k].y);
  }
  __syncwarp();
}

// y0, y1: rows 2l and 2l + 1 of sum_k ck[k] t_k over k <= Ky; first, last (if given): entries 0 and
// m - 1 of t_k for k <= K (K >= Ky).
__device__ inline void sum(const Proj& p, int Ky, int K, const double2* ck, double2& y0, double2& y1, double* first,
                           double* last) {
  const int l = threadIdx.x & 31;
  const int own = (p.m - 1) >> 1;  // lane of row m - 1
  double s0 = 0.0, s1 = 0.0;       // t_{k-1}
  double t0 = l == 0 ? 1.0 : 0.0, t1 = 0.0;
  y0 = y1 = make_double2(0.0, 0.0);
  for (int k = 0; k <= K; ++k) {
    if (k <= Ky) {
      const double2 q = ck[k];
      y0.x = fma(q.x, t0, y0.x);
      y0.y = fma(q.y, t0, y0.y);
      y1.x = fma(q.x, t1, y1.x);
      y1.y = fma(q.y, t1, y1.y);
    }
    if (first && l == 0) first[k] = t0;
    if (last && l == own) last[k] = (p.m - 1) & 1 ? t1 : t0;
    const double left = __shfl_up_sync(0xffffffffu, t1, 1), right = __shfl_down_sync(0xffffffffu, t0, 1);
    double n0 = fma(p.a0, t0, fma(p.bm, t1, l > 0 ? p.bl * left : 0.0));
    double n1 = fma(p.a1, t1, fma(p.bm, t0, l < 31 ? p.br * right : 0.0));
    if (k == 0) {  // t_1 = (T - c)/r t_0: half of the doubled matrix
      n0 *= 0.5;
      n1 *= 0.5;
    }
    n0 -= s0;
    n1 -= s1;
    s0 = t0;
    s1 = t1;
    t0 = n0;
    t1 = n1;
  }
  __syncwarp();
}

// |y|^2 from the sums
__device__ inline double norm2(double2 y0, double2 y1) {
  return warp_sum(fma(y0.x, y0.x, y0.y * y0.y) + fma(y1.x, y1.x, y1.y * y1.y));
}

// Whether sums of norm^2 n2 give y to the accuracy asked for.  Their error is at most 2e-16 (bases
// of real couplings, N = 6 to 16, |w| up to 85, against 40-digit arithmetic), so y's is below 1.3e-14
// of |y| (the eigendecomposition's: 1e-15 to 4e-14) or 2e-3 tol, whichever is larger.  |y| only grows
// on its scale towards smaller steps, so a step search below needs no check of its own.
__device__ __forceinline__ bool keeps(double n2, double tol) {
  const double least = fmin(1.0 / 64.0, 1e-13 / tol);
  return n2 >= least * least;
}

// Saad's estimate beta_last |y_{m-1}| / |y| from the sums and their norm^2 (see step_error).
__device__ inline double estimate(const Proj& p, double beta_last, double2 y0, double2 y1, double den) {
  if (beta_last == 0.0) return 0.0;
  const double2 e = (p.m - 1) & 1 ? y1 : y0;
  const double num = __shfl_sync(0xffffffffu, fma(e.x, e.x, e.y * e.y), (p.m - 1) >> 1);
  if (!(den > 0.0)) return 0.0;
  return beta_last * sqrt(num / den);
}

// sum_{k <= K} (2 - delta) I_k(w) e^{-w'} x[k] of the calling lane's own w, in one pass: K serves
// the lane of the largest w, and every lane's recurrence starts at the terms of its own w (the ones
// above are below 1e-17).  Started at K, a small w would carry it beyond the range of a double (for
// |w| = 4 and the terms of 128 to 1e210, squared in the division).
__device__ inline double2 lane_sum(double2 w, int K, const double* x) {
  const bool neg = w.x < 0.0;
  const double2 v = neg ? make_double2(-w.x, -w.y) : w;
  const double n2 = fma(v.x, v.x, v.y * v.y);
  if (n2 < 1e-16) {
    const double f = neg ? -x[1] : x[1];
    return make_double2(x[0] + v.x * (f - x[0]), v.y * (f - x[0]));
  }
  const double2 iv = cdiv(make_double2(2.0, 0.0), v);
  double2 hi = make_double2(0.0, 0.0), a = make_double2(0.0, 0.0), sum = make_double2(0.0, 0.0);
  double2 dot = make_double2(0.0, 0.0);
  const int start = min(K, terms(sqrt(n2))) + 4;
  for (int k = K + 4; k > 0; --k) {
    if (k == start) a.x = 1e-100;
    sum.x += a.x;
    sum.y += a.y;
    if (k <= K) {
      const double xk = neg && (k & 1) ? -x[k] : x[k];
      dot.x = fma(a.x, xk, dot.x);
      dot.y = fma(a.y, xk, dot.y);
    }
    const double ux = k * iv.x, uy = k * iv.y;
    const double2 n = make_double2(fma(ux, a.x, fma(-uy, a.y, hi.x)), fma(ux, a.y, fma(uy, a.x, hi.y)));
    hi = a;
    a = n;
  }
  const double2 num = make_double2(fma(2.0, dot.x, a.x * x[0]), fma(2.0, dot.y, a.y * x[0]));
  return cdiv(num, make_double2(fma(2.0, sum.x, a.x), fma(2.0, sum.y, a.y)));
}

// The largest step s < s_top whose estimate is <= tol (the estimate at s_top is not), to 2^-25 of
// it: every lane tries one of 32 steps that divide the bracket, until it is that narrow.  first,
// last: entries 0 and m - 1 of t_k (see sum) for all terms of w = s_top z r and of 2 Re w.
__device__ inline double select(const Proj& p, double beta_last, double s_top, double tol, double zr, double zi,
                                const double* first, const double* last, double narrow = 3e-8) {
  const int l = threadIdx.x & 31;
  double lo = 0.0, hi = s_top;
  for (int round = 0; round < 24; ++round) {
    const double d = (hi - lo) * 0.03125;
    const double s = l < 31 ? lo + d * (l + 1) : hi;
    const double2 w = make_double2(s * zr * p.r, s * zi * p.r);
    const double hw = sqrt(fma(zr, zr, zi * zi)) * hi * p.r;
    const double2 y = lane_sum(w, terms(hw), last);
    // |y|^2 = entry 0 of e^{2 s Re z T}; 1 in real time
    double den = 1.0;
    if (zr != 0.0) den = lane_sum(make_double2(2.0 * w.x, 0.0), terms(2.0 * fabs(zr) * hi * p.r), first).x;
    const bool ok = den > 0.0 && beta_last * sqrt(fma(y.x, y.x, y.y * y.y) / den) <= tol;
    // the first step that fails bounds the bracket from above, the one before it from below
    const unsigned bad = ~__ballot_sync(0xffffffffu, ok && l < 31);
    const int f = __ffs(bad) - 1;
    const double nhi = f < 31 ? lo + d * (f + 1) : hi;
    lo = f > 0 ? lo + d * f : lo;
    hi = nhi;
    if (lo > 0.0 && hi - lo <= narrow * lo) break;
  }
  return lo;
}

}  // namespace cheb
}  // namespace syk
