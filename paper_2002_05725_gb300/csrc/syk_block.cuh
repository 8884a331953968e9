// Row-block arithmetic of the complex64 matvec (syk_apply_block.cu), usable on the host too so
// that its index and sign algebra can be checked against the plain sum over masks on the CPU.
//
// The compact row index c splits, from the low end, into LB low bits, RB row bits, MB middle
// bits and the tile bits.  A thread owns the 2^RB rows that differ in the row bits, for ONE
// state.  Masks that agree outside the row bits form a coset: they read the same 2^RB partner
// rows, so a coset's partner rows are loaded into registers once and feed every mask of it.
// W, the popcount of a coset outside the row bits, fixes which row parts `lo` occur:
//   four-spin masks   |lo| = 4 - W, or 3 - W when the top spin n-1 is one of the four
//   two-spin masks    |lo| = 2 - W, or 1 - W with the top spin
//   the diagonal      W = 0, lo = 0
// so the five values of W give five bodies whose row pattern is known at compile time.
//
// Signs.  A Jordan-Wigner string puts Z on a spin s outside the mask's support when the number
// of support spins below s is odd.  Outside the row bits that is the same for every four-spin
// and two-spin mask of a coset (|lo| has the parity of W) and flips above the row bits when the
// top spin takes part (|lo| one less): zeta of the coset, plus the parity of the bits above for
// the masks with the top spin.  On a row bit it is (lo bits below) + lambda, lambda the popcount
// of the coset's low bits: the first is known at compile time, the second multiplies the rows
// of odd parity by (-1)^lambda once the support's share is folded into the tables.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <utility>

namespace syk {
namespace blk {

#define SYK_INLINE __attribute__((always_inline))
#define SYK_HD __host__ __device__ __forceinline__

constexpr int popc(uint32_t v) { return v ? int(v & 1u) + popc(v >> 1) : 0; }

// kind of the mask with row part lo in a coset of weight W
enum { kNone = 0, kM4 = 1, kM4Top = 2, kM2 = 3, kM2Top = 4 };
constexpr int mask_kind(int W, uint32_t lo) {
  return popc(lo) == 4 - W ? kM4 : popc(lo) == 3 - W ? kM4Top : popc(lo) == 2 - W ? kM2 : popc(lo) == 1 - W ? kM2Top : kNone;
}
// four-spin table entries of one mask: a value for each choice of its row support bits (and of
// the top spin's bit)
constexpr int mask_entries(int W, uint32_t lo) {
  return mask_kind(W, lo) == kM4 ? 1 << popc(lo) : mask_kind(W, lo) == kM4Top ? 2 << popc(lo) : 0;
}
constexpr int entries_before(int W, uint32_t lo) {
  int s = 0;
  for (uint32_t l = 0; l < lo; ++l) s += mask_entries(W, l);
  return s;
}
constexpr int coset_entries(int RB, int W) { return entries_before(W, 1u << RB); }
// A four-spin table entry holds the coefficient in both signs: (re, im), (-re, -im).
constexpr int kEntryBytes = 16;
// Two-spin tables of a mask, for each value u of its two support bits: sums of +-W_c over the
// bits outside the row, four bits at a time (16 values for each of ng groups), their sums over
// the row bits (2^RB values), then W_c of the RB row bits and of the top spin.
constexpr int kMaxGroups = 7;  // 31 compact bits less at least 3 row bits
constexpr int m2_values(int RB, int ng) { return 16 * ng + (1 << RB) + RB + 1; }
constexpr int m2_bytes(int RB, int ng) { return (4 * m2_values(RB, ng) * 8 + 15) / 16 * 16; }
// Bytes of a coset's tables: 2^W x entries, then for W = 2 the tables of its one two-spin mask.
// Two-spin masks with a support bit among the row bits or at the top spin (W < 2) are records of
// their own behind the cosets: many different row patterns, each of them rare.
constexpr int coset_bytes(int RB, int W, int ng) {
  return (coset_entries(RB, W) << W) * kEntryBytes + (W == 2 ? m2_bytes(RB, ng) : 0);
}
// Bytes that any one coset needs in a chunk: the header, its record and its tables.
constexpr int coset_most(int RB, int ng) {
  int m = m2_bytes(RB, ng);
  for (int W = 0; W <= 4; ++W) m = coset_bytes(RB, W, ng) > m ? coset_bytes(RB, W, ng) : m;
  return m + 32;
}
// bits of r at the set positions of lo, packed from the lowest
constexpr uint32_t pack_bits(uint32_t r, uint32_t lo) {
  uint32_t v = 0;
  int o = 0;
  for (int b = 0; b < 8; ++b)
    if ((lo >> b) & 1u) v |= ((r >> b) & 1u) << o++;
  return v;
}
// parity of r's bits outside lo that have an odd number of lo bits below them
constexpr bool row_sign(uint32_t r, uint32_t lo) {
  bool s = false;
  for (int b = 0; b < 8; ++b)
    if (((r >> b) & 1u) && !((lo >> b) & 1u) && (popc(lo & ((1u << b) - 1u)) & 1)) s = !s;
  return s;
}

// Two FP32 values in one 64-bit register pair; fma of both with one instruction.
typedef unsigned long long u64;
SYK_HD u64 pack2(float a, float b) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
#else
  union { float f[2]; u64 v; } u = {{a, b}};
  return u.v;
#endif
}
SYK_HD float2 unpack2(u64 v) {
#ifdef __CUDA_ARCH__
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
#else
  union { u64 v; float f[2]; } u = {v};
  return make_float2(u.f[0], u.f[1]);
#endif
}
SYK_HD void fma2(u64& a, u64 b, u64 c) {
#ifdef __CUDA_ARCH__
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a) : "l"(b), "l"(c));
#else
  const float2 x = unpack2(a), y = unpack2(b), z = unpack2(c);
  a = pack2(__builtin_fmaf(y.x, z.x, x.x), __builtin_fmaf(y.y, z.y, x.y));
#endif
}
SYK_HD float flip(float v, uint32_t sign) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(__float_as_uint(v) ^ sign);
#else
  return sign ? -v : v;
#endif
}

SYK_HD uint32_t parity(uint32_t v) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__popc(v) & 1u;
#else
  return (uint32_t)__builtin_popcount(v) & 1u;
#endif
}

// Compile-time loop: f(integral_constant<0>) ... f(integral_constant<N-1>).
template <typename F, int... I>
SYK_HD void static_for_impl(F&& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, typename F>
SYK_HD void static_for(F&& f) {
  static_for_impl(f, std::make_integer_sequence<int, N>{});
}

// Sums of a thread: y[r] = sum_m c (p.re, p.im) is kept as two packed sums, of the real and of
// the imaginary part of the coefficients times (p.re, p.im): y = re + i im.  Both operands of
// the packed multiply-add are then plain: no swapped or negated copy of the partner row.
template <int RB>
struct Acc {
  u64 re[1 << RB], im[1 << RB];
};

// What a thread needs to know of its rows, beside the pointers.
struct RowCtx {
  uint32_t x;       // compact index of the thread's row 0 (row bits clear)
  uint32_t xn;      // its bits outside the row bits, packed
  uint32_t q;       // top bit of row 0: sector ^ parity(x)
  uint32_t above;   // parity of x above the row bits
  int n;            // spins
  int LB;
  int ng;                   // groups of four of the bits outside the row
  const float* wd;          // diagonal couplings, n x n
  uint32_t B;               // states
  float2* share;            // the warp's scratch for two-spin coefficients (shared evaluation)
};

struct Coef {
  u64 re, im;  // (re, re), (im, im)
};
SYK_HD Coef load_coef(const unsigned char* a) {
  const float2 c = *reinterpret_cast<const float2*>(a);
  return {pack2(c.x, c.x), pack2(c.y, c.y)};
}
SYK_HD Coef negate(Coef c) {
  const float re = unpack2(c.re).x, im = unpack2(c.im).x;
  return {pack2(-re, -re), pack2(-im, -im)};
}

// whether any row of the class u needs the coefficient with parity class par and sign neg
constexpr bool needs(int RB, uint32_t lo, int u, int par, bool neg) {
  for (uint32_t r = 0; r < (1u << RB); ++r)
    if (int(pack_bits(r, lo)) == u && (par < 0 || (popc(r) & 1) == par) && row_sign(r, lo) == neg) return true;
  return false;
}

// One four-spin mask: every row r adds its coefficient times partner row r ^ LO.
// sg: sign bit of the coset for this thread.
template <int RB, int W, uint32_t LO>
SYK_HD void mask4(Acc<RB>& a, const u64 (&p)[1 << RB], const unsigned char* tab, const RowCtx& t, uint32_t sg) {
  constexpr int R = 1 << RB, K = popc(LO);
  constexpr bool top = mask_kind(W, LO) == kM4Top;
  if (top) sg ^= t.above;
  const unsigned char* T = tab + entries_before(W, LO) * kEntryBytes;
  static_for<(1 << K)>([&](auto ui) SYK_INLINE {
    constexpr int u = decltype(ui)::value;
    // with the top spin the rows of even and of odd parity have coefficients of their own
    static_for<(top ? 2 : 1)>([&](auto pi) SYK_INLINE {
      constexpr int par = top ? decltype(pi)::value : -1;
      const unsigned char* E = T + (top ? (2 * u + (t.q ^ (uint32_t)(par & 1))) : (uint32_t)u) * kEntryBytes;
      Coef pos = {}, neg = {};
      if constexpr (needs(RB, LO, u, par, false)) pos = load_coef(E + sg * 8u);
      if constexpr (needs(RB, LO, u, par, true))
        neg = needs(RB, LO, u, par, false) ? negate(pos) : load_coef(E + (sg ^ 1u) * 8u);
      static_for<R>([&](auto ri) SYK_INLINE {
        constexpr int r = decltype(ri)::value;
        if constexpr (int(pack_bits(r, LO)) == u && (par < 0 || (popc(r) & 1) == par)) {
          const Coef& c = row_sign(r, LO) ? neg : pos;
          fma2(a.re[r], c.re, p[r ^ LO]);
          fma2(a.im[r], c.im, p[r ^ LO]);
        }
      });
    });
  });
}

// The two-spin mask of a coset of weight 2: c(r) = (-1)^{zeta & x} sum_c (-1)^{x_c} W_c[u].  The
// sum over the bits outside the row comes from the tables, four bits a lookup; the row bits add
// their +-W_c in a binary tree over the rows, the top spin's sign being the rows' parity.
// un: bits of x at the coset's support.
template <int RB>
SYK_HD void mask2(Acc<RB>& a, const u64 (&p)[1 << RB], const unsigned char* tabs, const RowCtx& t, uint32_t un, uint32_t sg) {
  const float2* T = reinterpret_cast<const float2*>(tabs) + un * m2_values(RB, t.ng);
  const uint32_t s = sg << 31;
  float br = 0.f, bi = 0.f;
#pragma unroll 4
  for (int g = 0; g < t.ng; ++g) {
    const float2 w = T[16 * g + ((t.xn >> (4 * g)) & 15u)];
    br += w.x;
    bi += w.y;
  }
  br = flip(br, s);
  bi = flip(bi, s);
  const float2* Tr = T + 16 * t.ng + (1 << RB);
  // the highest row bit together with the top spin: for rows (that bit clear) of even and of odd
  // parity it adds +-(W + Wtop), +-(W - Wtop)
  const float2 wt0 = Tr[RB];
  const uint32_t st = s ^ (t.q << 31);
  const float2 wt = make_float2(flip(wt0.x, st), flip(wt0.y, st));
  float2 wr[RB];
#pragma unroll
  for (int b = 0; b < RB; ++b) {
    const float2 w = Tr[b];
    wr[b] = make_float2(flip(w.x, s), flip(w.y, s));
  }
  const float2 we = make_float2(wr[RB - 1].x + wt.x, wr[RB - 1].y + wt.y);
  const float2 wo = make_float2(wr[RB - 1].x - wt.x, wr[RB - 1].y - wt.y);
  static_for<(1 << RB)>([&](auto ri) SYK_INLINE {
    constexpr int r = decltype(ri)::value;
    float cr = br, ci = bi;
#pragma unroll
    for (int b = 0; b < RB - 1; ++b) {
      cr += ((r >> b) & 1) ? -wr[b].x : wr[b].x;
      ci += ((r >> b) & 1) ? -wr[b].y : wr[b].y;
    }
    constexpr bool up = (r >> (RB - 1)) & 1, odd = popc(r & ((1u << (RB - 1)) - 1u)) & 1;
    const float2 w = odd ? wo : we;
    cr += up ? -w.x : w.x;
    ci += up ? -w.y : w.y;
    fma2(a.re[r], pack2(cr, cr), p[r]);
    fma2(a.im[r], pack2(ci, ci), p[r]);
  });
}

// Coefficient of a two-spin record (x: row flip << 24 among the coset fields, y: zeta over the
// full spin index, z: its support spins a | b << 8) at row r of the thread.
template <int RB>
SYK_HD float2 m2_row(const uint4 rec, const unsigned char* tabs, const RowCtx& t, uint32_t r) {
  const uint32_t xf = t.x | (r << t.LB) | ((t.q ^ parity(r)) << (t.n - 1));
  const uint32_t u = ((xf >> (rec.z & 31u)) & 1u) | (((xf >> ((rec.z >> 8) & 31u)) & 1u) << 1);
  const float2* T = reinterpret_cast<const float2*>(tabs) + u * m2_values(RB, t.ng);
  float2 c = T[16 * t.ng + r];
#pragma unroll
  for (int g = 0; g < kMaxGroups; ++g)
    if (g < t.ng) {
      const float2 w = T[16 * g + ((t.xn >> (4 * g)) & 15u)];
      c.x += w.x;
      c.y += w.y;
    }
  const float2 w = T[16 * t.ng + (1 << RB) + RB];
  const uint32_t st = (xf >> (t.n - 1)) << 31, s = parity(rec.y & xf) << 31;
  return make_float2(flip(c.x + flip(w.x, st), s), flip(c.y + flip(w.y, st), s));
}

#ifdef __CUDACC__
// The two-spin mask of a coset of weight 2 for 8 or 16 states, whose threads of a row block are B
// neighbouring lanes: each lane evaluates 2^RB / B of the rows from the tables and the lanes
// exchange them through the warp's scratch, so that a row's coefficient is computed once and not
// once a state.  m2_share writes the scratch (before the partner rows take their registers),
// m2_apply uses it.
constexpr int kShareStride = 2;  // float2 of padding between the row blocks of a warp
constexpr int share_bytes(int RB, int B) { return 32 / B * ((1 << RB) + kShareStride) * 8; }
template <int RB>
__device__ __forceinline__ float2* m2_share(const unsigned char* tabs, const RowCtx& t, uint32_t un, uint32_t sg) {
  constexpr int R = 1 << RB;
  const uint32_t lane = threadIdx.x & 31u, B = t.B;
  float2* blk = t.share + (lane / B) * (R + kShareStride);
  const float2* T = reinterpret_cast<const float2*>(tabs) + un * m2_values(RB, t.ng);
  float2 base = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int g = 0; g < t.ng; ++g) {
    const float2 w = T[16 * g + ((t.xn >> (4 * g)) & 15u)];
    base.x += w.x;
    base.y += w.y;
  }
  const float2 w = T[16 * t.ng + R + RB];
  const uint32_t s = sg << 31;
  __syncwarp();  // the previous mask's values have been read
#pragma unroll 1
  for (uint32_t r = lane & (B - 1u); r < (uint32_t)R; r += B) {
    const float2 c = T[16 * t.ng + r];
    const uint32_t st = (t.q ^ parity(r)) << 31;
    blk[r] = make_float2(flip(base.x + c.x + flip(w.x, st), s), flip(base.y + c.y + flip(w.y, st), s));
  }
  __syncwarp();
  return blk;
}
template <int RB>
__device__ __forceinline__ void m2_apply(Acc<RB>& a, const u64 (&p)[1 << RB], const float2* blk) {
  static_for<(1 << RB) / 2>([&](auto hi) SYK_INLINE {
    constexpr int r = 2 * decltype(hi)::value;
    const float4 c = *reinterpret_cast<const float4*>(blk + r);
    fma2(a.re[r], pack2(c.x, c.x), p[r]);
    fma2(a.im[r], pack2(c.y, c.y), p[r]);
    fma2(a.re[r + 1], pack2(c.z, c.z), p[r + 1]);
    fma2(a.im[r + 1], pack2(c.w, c.w), p[r + 1]);
  });
}
// The same for a two-spin record of its own (see m2_row).
template <int RB>
__device__ __forceinline__ float2* m2_share_record(const uint4 rec, const unsigned char* tabs, const RowCtx& t) {
  constexpr int R = 1 << RB;
  const uint32_t lane = threadIdx.x & 31u, B = t.B;
  float2* blk = t.share + (lane / B) * (R + kShareStride);
  __syncwarp();
  if constexpr (R >= 32) {  // two rows at a time
#pragma unroll 1
    for (uint32_t r = lane & (B - 1u); r < (uint32_t)R; r += 2 * B) {
      const float2 c0 = m2_row<RB>(rec, tabs, t, r), c1 = m2_row<RB>(rec, tabs, t, r + B);
      blk[r] = c0;
      blk[r + B] = c1;
    }
  } else {
#pragma unroll 1
    for (uint32_t r = lane & (B - 1u); r < (uint32_t)R; r += B) blk[r] = m2_row<RB>(rec, tabs, t, r);
  }
  __syncwarp();
  return blk;
}
#endif

// One two-spin record: row r adds its coefficient times partner row r ^ lo.
template <int RB, bool SHARE>
SYK_HD void m2_record(Acc<RB>& a, const unsigned char* prow, int stride, const uint4 rec, const unsigned char* tabs,
                      const RowCtx& t) {
  constexpr int R = 1 << RB;
  const uint32_t lo = (rec.x >> 24) & 0x1fu;
#ifdef __CUDA_ARCH__
  if constexpr (SHARE) {
    const float2* blk = m2_share_record<RB>(rec, tabs, t);
    u64 p[R];
#pragma unroll
    for (int r = 0; r < R; ++r) p[r] = *reinterpret_cast<const u64*>(prow + ((uint32_t)r ^ lo) * stride);
    m2_apply<RB>(a, p, blk);
    return;
  }
#endif
  static_for<R>([&](auto ri) SYK_INLINE {
    constexpr int r = decltype(ri)::value;
    const u64 p = *reinterpret_cast<const u64*>(prow + ((uint32_t)r ^ lo) * stride);
    const float2 c = m2_row<RB>(rec, tabs, t, r);
    fma2(a.re[r], pack2(c.x, c.x), p);
    fma2(a.im[r], pack2(c.y, c.y), p);
  });
}

// The diagonal: sum_{c<d} w_cd (-1)^{x_c + x_d}, split into the part outside the row bits, the
// row bits' linear terms and the pairs among row bits and the top spin.
template <int RB>
SYK_HD void diagonal(Acc<RB>& a, const u64 (&p)[1 << RB], const RowCtx& t) {
  const int n = t.n, top = n - 1, r0 = t.LB;
  auto w = [&](int c, int d) { return c < d ? t.wd[c * n + d] : t.wd[d * n + c]; };
  auto outside = [&](int c) { return c < r0 || c >= r0 + RB; };
  float q0 = 0.f, lt = 0.f, lb[RB] = {};
  for (int c = 0; c < top; ++c) {
    if (!outside(c)) continue;
    const uint32_t sc = ((t.x >> c) & 1u) << 31;
    float in = 0.f;
    for (int d = c + 1; d < top; ++d)
      if (outside(d)) in += flip(t.wd[c * n + d], ((t.x >> d) & 1u) << 31);
    q0 += flip(in, sc);
    lt += flip(t.wd[c * n + top], sc);
    for (int b = 0; b < RB; ++b) lb[b] += flip(w(c, r0 + b), sc);
  }
  static_for<(1 << RB)>([&](auto ri) SYK_INLINE {
    constexpr int r = decltype(ri)::value;
    const uint32_t st = ((t.q ^ (popc(r) & 1)) & 1u) << 31;
    float v = q0 + flip(lt, st);
#pragma unroll
    for (int b = 0; b < RB; ++b) {
      float in = lb[b] + flip(t.wd[(r0 + b) * n + top], st);
#pragma unroll
      for (int d = b + 1; d < RB; ++d) in += ((r >> d) & 1) ? -t.wd[(r0 + b) * n + r0 + d] : t.wd[(r0 + b) * n + r0 + d];
      v += ((r >> b) & 1) ? -in : in;
    }
    fma2(a.re[r], pack2(v, v), p[r]);
  });
}

// Record of a coset, in front of its tables.
//   x: middle-bit flip | low-bit flip << 16 | (low bits' popcount odd) << 31
//   y: zeta (compact bits outside the row bits)
//   z: right shifts that bring support bit k of x to bit k (a byte each; 31: none)
//   w: byte offset of its tables in the chunk
SYK_HD uint32_t support(uint32_t x, uint32_t s) {
  return ((x >> (s & 31u)) & 1u) | ((x >> ((s >> 8) & 31u)) & 2u) | ((x >> ((s >> 16) & 31u)) & 4u) |
         ((x >> ((s >> 24) & 31u)) & 8u);
}
// What a thread derives from a coset's record; computed one coset ahead of its use.
struct CosetAt {
  const unsigned char* prow;  // the thread's partner row 0 in the staged tile
  const unsigned char* tb;    // the coset's tables
  uint32_t un, sg;            // bits of x at its support, sign bit of zeta & x
  uint32_t odd;               // whether the popcount of its low bits is odd
};

// One coset of weight W.  stride: bytes between partner rows.  LOWS: there are low bits, whose
// odd popcount flips the rows of odd parity: done on the partner rows, as partner row r ^ lo
// feeds row r and |lo|'s parity is in the tables.
template <int RB, int W, bool LOWS, bool SHARE = false>
SYK_HD void coset(Acc<RB>& a, const CosetAt& k, int stride, const RowCtx& t) {
  constexpr int R = 1 << RB;
#ifdef __CUDA_ARCH__
  const float2* shared = nullptr;
  if constexpr (SHARE && W == 2)
    shared = m2_share<RB>(k.tb + (coset_entries(RB, W) << W) * kEntryBytes, t, k.un, k.sg);
#endif
  u64 p[R];
#pragma unroll
  for (int r = 0; r < R; ++r) p[r] = *reinterpret_cast<const u64*>(k.prow + r * stride);
  if (LOWS) {
    const u64 f = k.odd ? 0x8000000080000000ull : 0ull;
    static_for<R>([&](auto ri) SYK_INLINE {
      constexpr int r = decltype(ri)::value;
      if constexpr (popc(r) & 1) p[r] ^= f;
    });
  }
  const uint32_t un = k.un, sg = k.sg;
  const unsigned char* tb = k.tb;
  const unsigned char* tab = tb + un * (coset_entries(RB, W) * kEntryBytes);
  static_for<R>([&](auto l) SYK_INLINE {
    constexpr uint32_t LO = decltype(l)::value;
    constexpr int kind = mask_kind(W, LO);
    if constexpr (kind == kM4 || kind == kM4Top) mask4<RB, W, LO>(a, p, tab, t, sg);
  });
#ifdef __CUDA_ARCH__
  if constexpr (SHARE && W == 2) {
    m2_apply<RB>(a, p, shared);
  } else
#endif
  if constexpr (W == 2) {
    mask2<RB>(a, p, tb + (coset_entries(RB, W) << W) * kEntryBytes, t, un, sg);
  }
  if constexpr (W == 0) diagonal<RB>(a, p, t);
}

}  // namespace blk
}  // namespace syk
