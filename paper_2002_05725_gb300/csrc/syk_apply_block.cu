// Row-block matvec (see syk_block_kernel.cuh): its launch rule, and its kernels with 8 rows per
// thread for small sectors.
#include "syk_block_kernel.cuh"

namespace syk {
namespace {

bool pow2(int64_t v) { return (v & (v - 1)) == 0; }

// Low bits of a row-block launch: a row slot of B << lb elements is 16 for 1 to 16 states in
// powers of two, so that a half warp reads 128 contiguous bytes, and at most 24 otherwise.
int low_bits(int64_t B) {
  int lb = 0;
  while ((B << (lb + 1)) <= (pow2(B) ? 16 : 24)) ++lb;
  return lb;
}

}  // namespace

int block_aux(int n, int rb, bool df) {
  const int ng = (n - 1 - rb + 3) / 4;
  return df ? blk::df_coset_most(3, ng) : rb == 5 ? blk::coset_most(5, ng) : blk::coset_most(3, ng);
}

size_t block_smem(int64_t B, int lb, int rb, int mb, int auxb, int elem) {
  const size_t warps = ((size_t(B) << (lb + mb)) + 31) / 32;
  const bool df = elem == 16;
  size_t share = 0;
  if (B == 8 || B == 16) share = warps * (rb == 5 ? blk::share_bytes(5, int(B)) : blk::share_bytes(3, int(B)));
  return (df ? 2 : 3) * ((size_t(B) << (lb + rb + mb)) * elem + auxb) + 64 + share;
}

bool block_shape(int n, int64_t batch, int dtype, int rb, int mb, int cs, BlockShape* sh) {
  const bool df = dtype == SYK_C128;
  if (batch < 1 || batch > 32 || mb < 0 || (rb != 3 && rb != 5) || (df && (rb != 3 || !pow2(batch) || batch > 16))) return false;
  *sh = {rb, low_bits(batch), mb, cs, block_aux(n, rb, df), df};
  const int tb = sh->lb + rb + mb;
  const int64_t D = int64_t(1) << (n - 1);
  return tb <= n - 1 && (batch << (sh->lb + mb)) <= 256 && (D >> tb) * cs <= ep_capacity(D) &&
         block_smem(batch, sh->lb, rb, mb, sh->auxb, df ? 16 : 8) <= kMaxSmemPerCta;
}

bool block_default(int n, int64_t batch, int dtype, BlockShape* sh) {
  if (batch < 1 || batch > 32 || n - 1 > 31) return false;
  const int64_t D = int64_t(1) << (n - 1);
  if (dtype == SYK_C128) {
    // One state, and 2 and 4 states of sectors up to 2^15 elements: there the tiled double-float
    // kernel is bound by latency (N = 28: 1 state 337 us, 140 here, 2 states 298 and 156, 4 states 255
    // and 163; N = 36, 1 state 1.94 and 1.32 ms; N = 40, 1 state 7.7 and 6.8).  Beyond it is bound by
    // the FP32 operations that both do and its smaller code wins (N = 36, 2 states 2.28 ms, 2.45 here;
    // 4 states 3.9 and 4.7, 16 states 13.0 and 17.0).  The line lies on the safe side: with the best of
    // its shapes this kernel is the faster one up to 2^17 elements (N = 30, 4 states 419 us tiled and
    // 332 here; N = 32, 2 states 671 and 412, 4 states 828 and 756; N = 34, 2 states 1.26 and 1.05 ms),
    // at 2^18 no more (N = 34, 4 states 1.89 and 1.96 ms).
    if (batch != 1 && !((batch == 2 || batch == 4) && D * batch <= (int64_t(1) << 15))) return false;
    const int full = 4;  // 256 threads
    const int64_t ctas = 2 * int64_t(sm_count()), tiles = (D * batch) >> (4 + 3 + full);
    int cs = 1, mb = full;
    while (cs < 8 && tiles * cs * 2 <= ctas) cs *= 2;
    if (cs == 8) mb = 3;
    for (; mb >= 0; --mb)
      if (block_shape(n, batch, dtype, 3, mb, cs, sh)) return true;
    return false;
  }
  // State counts that are no power of two stay with the row kernel in sectors below 2^10.  That is not
  // for speed (N = 20: 3 states 256 us there and 15 here, 6 states 266 and 15; N = 12, 6 states 46 and
  // 16): a process whose staged copies time out still has a matvec without waits, which the failure
  // tests ask for with 3 states at N = 20.  (N = 24, 6 states, beyond the line: 496 and 21 us.)
  if (!pow2(batch) && D < 1024) return false;
  const int lb = low_bits(batch);
  int full = 0;  // middle bits of a 256-thread CTA
  while ((batch << (lb + full + 1)) <= 256) ++full;
  // 32 rows per thread above 2^16 elements, 8 rows below: there the larger number of threads
  // counts (N = 32, 1 state: 45 us with 8 rows, 63 with 32; N = 28, 8 states: 39 both; N = 28, 16
  // states: 68 and 60; N = 38, 8 states: 2.9 and 1.9 ms).  Full tiles (256 threads, one CTA per
  // SM) halve the copies of 128-thread ones (N = 40, 16 states: 8.7 against 13.7 ms); a cluster
  // splits a tile's chunks while that leaves at most about one CTA per SM (N = 32, 16 states, 64
  // tiles: 248 us with 2 CTAs a tile, 459 with 1; N = 38, 8 states, 256 tiles: 1.97 ms with 1, 2.01
  // with 2).  Clusters of 8 only with small CTAs, several to an SM.
  // 4, 8 and 16 states take more: each CTA of a cluster sums a share of the masks, and shorter FP32
  // chains keep the rounding error below that of the coset kernel, whose clusters were of 4 or 8
  // there.  Relative error (2-norm) of that one, with the rule above and with this one, and the time
  // it takes: N = 32, 16 states 4.1e-7, 5.4e-7, 3.8e-7, 248 -> 258 us; N = 34, 8 states 4.6e-7, 6.1e-7,
  // 4.3e-7, 320 -> 332 us; N = 36, 4 states 5.2e-7, 6.9e-7, 4.9e-7, 451 -> 474 us; N = 38, 4 states
  // 8.3e-7, 1.1e-6, 7.7e-7, 1.08 -> 1.09 ms.  Where a tile has one CTA, launch_apply_block sums in parts.
  if (D * batch > (int64_t(1) << 16)) {
    const int64_t tiles = D >> std::min(n - 1, lb + 5 + full);
    const int mb = tiles >= 25 ? full : full - 1;
    int cs = tiles >= 100 ? 1 : tiles >= 50 ? 2 : 4;
    if (cs == 2 && (batch == 4 || batch == 8 || batch == 16)) cs = 4;
    if (cs == 1 && batch == 4 && tiles < 200) cs = 2;
    if (block_shape(n, batch, dtype, 5, mb, cs, sh)) return true;
  }
  for (int mb = std::min(3, full); mb >= 0; --mb)
    if (block_shape(n, batch, dtype, 3, mb, 8, sh)) return true;
  return false;
}

int launch_apply_block(const ApplyParams& p, int64_t batch, const void* psi, void* y, cudaStream_t st, BlockShape sh) {
  if (reinterpret_cast<uintptr_t>(psi) & 15) return 1;  // bulk copies start on 16-byte boundaries
  BlockArgs a = {};
  a.B = (int)batch;
  a.LB = sh.lb;
  a.MB = sh.mb;
  a.SE = a.B << sh.lb;
  a.nt = a.SE << sh.mb;
  a.auxb = sh.auxb;
  const BlockLayout* L = nullptr;
  int lr = block_layout(p.terms, sh.rb, sh.lb, sh.mb, sh.cs, sh.auxb, sh.df, false, false, &L);
  if (lr > 0 && !p.no_alloc) {
    // The first launch of a shape builds its layout, under capture too: the kernels that would stand
    // in have layouts of their own, which nothing builds any more where this kernel is the default.
    // (The query fails on the legacy stream while another one is under capture: then the former
    // kernels take over, as far as they can.)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) cudaGetLastError();
    else
      lr = block_layout(p.terms, sh.rb, sh.lb, sh.mb, sh.cs, sh.auxb, sh.df, true, cap != cudaStreamCaptureStatusNone, &L);
  }
  if (lr != SYK_OK) return lr > 0 ? 1 : lr;
  for (int k = 0; k < 9; ++k) a.begin[k] = L->begin[k];
  const int which = a.SE != 16 ? kBlockAny : sh.lb == 0 ? kBlock16 : batch == 8 ? kBlockShare : kBlockPow2;
  const bool share = which == kBlock16 || which == kBlockShare;
  if (sh.df) return launch_block_df(p, a, sh.cs, L, psi, y, st);
  // 8 and 16 states with one CTA a tile: in parts up to the size where the coset kernel still split a
  // row over 4 CTAs or more (from N = 38, 16 states, and N = 40, 8 states, on one chain is no worse
  // than it was: 1.11e-6 against 1.17e-6, 1.22e-6 against 1.30e-6)
  if (sh.rb == 5 && share && sh.cs == 1 && p.D * batch < (int64_t(1) << 22)) {
    a.part = (a.begin[1] + 7) / 8;
    return launch_block32_parts(p, a, which, L, psi, y, st);
  }
  if (sh.rb == 5)
    return share ? launch_block32_share(p, a, which, sh.cs, L, psi, y, st)
                 : launch_block32_direct(p, a, which, sh.cs, L, psi, y, st);
  return share                 ? launch_block<BlockF32, 3, 16, true, true, 256, 1>(p, a, sh.cs, L, psi, y, st)
         : which == kBlockPow2 ? launch_block<BlockF32, 3, 16, true, false, 256, 1>(p, a, sh.cs, L, psi, y, st)
                               : launch_block<BlockF32, 3, 0, true, false, 256, 1>(p, a, sh.cs, L, psi, y, st);
}

}  // namespace syk
