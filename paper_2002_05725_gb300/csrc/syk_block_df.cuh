// Row-block arithmetic of the complex128 matvec in double-float form (syk_df.cuh) on the layout of
// syk_block.cuh: 8 rows per thread, each a (re_hi, im_hi, re_lo, im_lo) sum.
//
// 48 FP32 operations per row and mask leave coefficients and partner rows cheap, so every two-spin
// mask is a record of its own here, and 8 rows (32 registers of sums, 32 of partner rows) let 16
// warps share an SM.  The sums are renormalised after every coset (of weight 4, one mask a row:
// every eighth), as the tiled kernel does after 16 masks.
#pragma once
#include "syk_block.cuh"
#ifdef __CUDACC__
#include "syk_df.cuh"
#endif

namespace syk {
namespace blk {

// A four-spin entry: the coefficient as a double-float complex value, and its negative.
constexpr int kDfEntryBytes = 32;
constexpr int df_m2_bytes(int RB, int ng) { return 4 * m2_values(RB, ng) * 16; }
constexpr int df_coset_bytes(int RB, int W) { return (coset_entries(RB, W) << W) * kDfEntryBytes; }
constexpr int df_coset_most(int RB, int ng) {
  int m = df_m2_bytes(RB, ng);
  for (int W = 0; W <= 4; ++W) m = df_coset_bytes(RB, W) > m ? df_coset_bytes(RB, W) : m;
  return m + 32;
}

#ifdef __CUDACC__
template <int RB>
struct AccDf {
  float4 v[1 << RB];
};

__device__ __forceinline__ float4 neg4(float4 a) { return make_float4(-a.x, -a.y, -a.z, -a.w); }
__device__ __forceinline__ float4 flip4(float4 a, uint32_t s) {
  return make_float4(flip(a.x, s), flip(a.y, s), flip(a.z, s), flip(a.w, s));
}
template <int RB>
__device__ __forceinline__ void renorm(AccDf<RB>& a) {
#pragma unroll
  for (int r = 0; r < (1 << RB); ++r) df_renorm4(a.v[r]);
}

template <int RB, int W, uint32_t LO>
__device__ __forceinline__ void mask4_df(AccDf<RB>& a, const float4 (&p)[1 << RB], const unsigned char* tab, const RowCtx& t,
                                         uint32_t sg) {
  constexpr int R = 1 << RB, K = popc(LO);
  constexpr bool top = mask_kind(W, LO) == kM4Top;
  if (top) sg ^= t.above;
  const unsigned char* T = tab + entries_before(W, LO) * kDfEntryBytes;
  static_for<(1 << K)>([&](auto ui) SYK_INLINE {
    constexpr int u = decltype(ui)::value;
    static_for<(top ? 2 : 1)>([&](auto pi) SYK_INLINE {
      constexpr int par = top ? decltype(pi)::value : -1;
      const unsigned char* E = T + (top ? (2 * u + (t.q ^ (uint32_t)(par & 1))) : (uint32_t)u) * kDfEntryBytes;
      const float4 c = *reinterpret_cast<const float4*>(E + sg * 16u);
      static_for<R>([&](auto ri) SYK_INLINE {
        constexpr int r = decltype(ri)::value;
        if constexpr (int(pack_bits(r, LO)) == u && (par < 0 || (popc(r) & 1) == par))
          df_cmac(a.v[r], row_sign(r, LO) ? neg4(c) : c, p[r ^ LO]);
      });
    });
  });
}

// Coefficient of a two-spin record at row r (see m2_row), in double-float.
template <int RB>
__device__ __forceinline__ float4 m2_row_df(const uint4 rec, const unsigned char* tabs, const RowCtx& t, uint32_t r) {
  const uint32_t xf = t.x | (r << t.LB) | ((t.q ^ parity(r)) << (t.n - 1));
  const uint32_t u = ((xf >> (rec.z & 31u)) & 1u) | (((xf >> ((rec.z >> 8) & 31u)) & 1u) << 1);
  const float4* T = reinterpret_cast<const float4*>(tabs) + u * m2_values(RB, t.ng);
  float4 c = T[16 * t.ng + r];
#pragma unroll 1
  for (int g = 0; g < t.ng; ++g) {
    const float4 w = T[16 * g + ((t.xn >> (4 * g)) & 15u)];
    df_add_signed(c.x, c.z, w.x, w.z, false);
    df_add_signed(c.y, c.w, w.y, w.w, false);
  }
  const float4 w = T[16 * t.ng + (1 << RB) + RB];
  const bool top = (xf >> (t.n - 1)) & 1u;
  df_add_signed(c.x, c.z, w.x, w.z, top);
  df_add_signed(c.y, c.w, w.y, w.w, top);
  df_renorm4(c);
  return flip4(c, parity(rec.y & xf) << 31);
}

template <int RB>
__device__ __forceinline__ void m2_record_df(AccDf<RB>& a, const unsigned char* prow, int stride, const uint4 rec,
                                             const unsigned char* tabs, const RowCtx& t) {
  const uint32_t lo = (rec.x >> 24) & 0x1fu;
#pragma unroll
  for (int r = 0; r < (1 << RB); ++r)
    df_cmac(a.v[r], m2_row_df<RB>(rec, tabs, t, r), *reinterpret_cast<const float4*>(prow + ((uint32_t)r ^ lo) * stride));
}

// The diagonal of a row in double-float (wd: n x n (hi, lo) pairs)
__device__ __forceinline__ float4 diag_df(const float2* __restrict__ wd, int n, uint32_t xf) {
  float hi = 0.f, lo = 0.f;
  for (int c = 0; c < n - 1; ++c)
    for (int d = c + 1; d < n; ++d) {
      const float2 w = __ldg(&wd[c * n + d]);
      df_add_signed(hi, lo, w.x, w.y, ((xf >> c) ^ (xf >> d)) & 1u);
    }
  df_renorm(hi, lo);
  return make_float4(hi, 0.f, lo, 0.f);
}

template <int RB, int W, bool LOWS>
__device__ __forceinline__ void coset_df(AccDf<RB>& a, const CosetAt& k, int stride, const RowCtx& t, const float2* wd) {
  constexpr int R = 1 << RB;
  float4 p[R];
#pragma unroll
  for (int r = 0; r < R; ++r) p[r] = *reinterpret_cast<const float4*>(k.prow + r * stride);
  if constexpr (W == 0) {
#pragma unroll
    for (int r = 0; r < R; ++r)
      df_cmac(a.v[r], diag_df(wd, t.n, t.x | ((uint32_t)r << t.LB) | ((t.q ^ parity(r)) << (t.n - 1))), p[r]);
  }
  if (LOWS) {
    const uint32_t f = k.odd << 31;
    static_for<R>([&](auto ri) SYK_INLINE {
      constexpr int r = decltype(ri)::value;
      if constexpr (popc(r) & 1) p[r] = flip4(p[r], f);
    });
  }
  const unsigned char* tab = k.tb + k.un * (coset_entries(RB, W) * kDfEntryBytes);
  static_for<R>([&](auto l) SYK_INLINE {
    constexpr uint32_t LO = decltype(l)::value;
    constexpr int kind = mask_kind(W, LO);
    if constexpr (kind == kM4 || kind == kM4Top) mask4_df<RB, W, LO>(a, p, tab, t, k.sg);
  });
}
#endif

}  // namespace blk
}  // namespace syk
