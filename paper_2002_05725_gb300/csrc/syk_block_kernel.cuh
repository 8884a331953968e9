// K1 variant: y = H psi in one parity sector (Supp. Sec. I.B), with the rows of a thread taken as a
// block of 2^RB rows (syk_block.cuh): complex64 (BlockF32), complex128 in double-float arithmetic
// (BlockDf, 8 rows; its figures stand in syk_block_df.cuh).  What follows is for complex64.
//
// A CTA owns a tile of 2^(LB+RB+MB) rows of all B states; thread t = (mid, low, state) owns the
// 2^RB rows between its low and middle bits, for one state.  Per tile flip h the partner tile
// psi[tile ^ h] and the chunk's coset records and tables come into shared memory by bulk
// asynchronous copies, in a ring of kStages stages; the warp that is last to finish a chunk
// refills its stage, so warps may run ahead of one another by the depth of the ring.
//
// Why this split.  The matvec is 8 flop per nonzero and state on operands in shared memory; a
// thread with one row and all states reads a partner row anew for every mask (or for 1.2 masks,
// k_apply_coset<16, 1>) and is bound by the shared-memory port.  Here a partner row read once
// feeds on average 3.4 masks (N = 40), and one coefficient lookup feeds all rows of a thread that
// share it.  The multiply-adds are the packed two-wide FP32 form: the same FP32 rate (measured
// 79.3 against 70.7 TFLOP/s in a register-only loop) for half the issue slots, which the
// coefficient work then takes.  256 threads of 255 registers fill an SM: 128 registers of sums,
// 64 of partner rows.  Bound now (N = 38, 16 states): FP32 pipe 54 % of its cycles, the rest
// latency with 2 warps a scheduler; shared-memory port 32 %, L2 14 %.  Without the copies the
// kernel takes as long, without the cosets of weight 4 (one mask a row: 512 cycles of the port
// against 256 of the FP32 pipe) 20 % less.
// Measured (GB300, per matvec, before -> after; before: the faster of the coset, tiled,
// one-state and row kernels' defaults): N = 40, 16 states 10.45 -> 8.44 ms (40 TFLOP/s); N = 48,
// 1 state 59.1 -> 19.1 ms; N = 36, 8 states 1.70 -> 0.80 ms; N = 34, 6 states 2.28 -> 0.39 ms;
// N = 32, 16 states 408 -> 258 us; N = 28, 8 states 136 -> 42 us, 1 state 328 -> 27 us; N = 20, 8
// states 69 -> 16 us.  Errors against 64-bit sums are 0.5 to 0.95 of the former kernels' for 1, 2, 4,
// 8 and 16 states, N = 20 to 42 (one rounding per product-sum instead of two, but longer chains: see
// PARTS), and 0.25 to 0.65 of the row kernel's for other counts.
// Tried and slower: 16 rows per thread with twice the threads (9.1 against 8.7 ms at N = 40, more
// shared-memory reads per mask); coefficients stored ready-paired (wider reads cost the port more
// than the register moves they save); two-spin coefficients per thread instead of per row block
// (9.4 against 8.7 ms); half the warps taking the cosets in another order (9.3, register spills).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "syk_block.cuh"
#include "syk_block_df.cuh"
#include "syk_tile.cuh"

namespace syk {

struct BlockArgs {
  int B, LB, MB;
  int SE;        // elements per row slot: B << LB
  int nt;        // threads that own rows: SE << MB
  int auxb;      // bytes of a stage for a chunk's records and tables
  int part;      // PARTS: chunks after which the sums so far go to y
  int begin[9];  // chunk range of each CTA of a tile
};

// What the kernel does per arithmetic: complex64 with packed FP32 sums, complex128 in double-float.
template <int RB, bool SHARE>
struct BlockF32 {
  using Out = float2;
  using Sum = float2;
  using Acc = blk::Acc<RB>;
  static constexpr int kElem = 8, kRing = 3;
  static __device__ __forceinline__ void zero(Acc& a) {
#pragma unroll
    for (int r = 0; r < (1 << RB); ++r) a.re[r] = a.im[r] = 0ull;
  }
  template <int W, bool LOWS>
  static __device__ __forceinline__ void coset(Acc& a, const blk::CosetAt& at, int stride, const blk::RowCtx& t,
                                               const ApplyParams&) {
    blk::coset<RB, W, LOWS, SHARE>(a, at, stride, t);
  }
  static __device__ __forceinline__ void record(Acc& a, const unsigned char* prow, int stride, const uint4 rec,
                                                const unsigned char* tabs, const blk::RowCtx& t) {
    blk::m2_record<RB, SHARE>(a, prow, stride, rec, tabs, t);
  }
  static __device__ __forceinline__ void renorm(Acc&) {}
  static __device__ __forceinline__ Sum get(const Acc& a, int r) {
    const float2 x = blk::unpack2(a.re[r]), y = blk::unpack2(a.im[r]);
    return make_float2(x.x - y.y, x.y + y.x);
  }
  static __device__ __forceinline__ void add(Sum& a, const Sum b) {
    a.x += b.x;
    a.y += b.y;
  }
  static constexpr int share(int B) { return blk::share_bytes(RB, B); }
};
template <int RB, bool SHARE>
struct BlockDf {
  using Out = double2;
  using Sum = double2;
  using Acc = blk::AccDf<RB>;
  static constexpr int kElem = 16, kRing = 2;
  static __device__ __forceinline__ void zero(Acc& a) {
#pragma unroll
    for (int r = 0; r < (1 << RB); ++r) a.v[r] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  template <int W, bool LOWS>
  static __device__ __forceinline__ void coset(Acc& a, const blk::CosetAt& at, int stride, const blk::RowCtx& t,
                                               const ApplyParams& p) {
    blk::coset_df<RB, W, LOWS>(a, at, stride, t, p.wd_df);
    if (W < 4) blk::renorm(a);
  }
  static __device__ __forceinline__ void record(Acc& a, const unsigned char* prow, int stride, const uint4 rec,
                                                const unsigned char* tabs, const blk::RowCtx& t) {
    blk::m2_record_df<RB>(a, prow, stride, rec, tabs, t);
    blk::renorm(a);
  }
  static __device__ __forceinline__ void renorm(Acc& a) { blk::renorm(a); }
  static __device__ __forceinline__ Sum get(const Acc& a, int r) { return df_to_double2(a.v[r]); }
  static __device__ __forceinline__ void add(Sum& a, const Sum b) {
    a.x += b.x;
    a.y += b.y;
  }
  static constexpr int share(int) { return 0; }
};
// an element of a CTA of the cluster (8-byte words)
template <typename T>
__device__ __forceinline__ T ld_cluster_elem(uint32_t a) {
  T v;
  unsigned long long* w = reinterpret_cast<unsigned long long*>(&v);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(T) / 8); ++i)
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(w[i]) : "r"(a + 8u * i) : "memory");
  return v;
}

// SEC: SE when known at compile time (16), so that row offsets are immediates; 0 otherwise.
// PARTS: a row's sum is taken in eight parts, added up in y.  In one FP32 chain its rounding error grows
// with the number of masks, and where the kernels before this one split a row over 4 or 8 CTAs of a
// cluster, one chain was worse than they were (launch_apply_block says where that is).  Relative error
// (2-norm) of the former kernels, of one chain and of the parts, and the time of the latter two:
// N = 34, 16 states 4.6e-7, 8.6e-7, 3.6e-7, 595 -> 600 us; N = 36, 8 states 5.2e-7, 9.7e-7, 3.9e-7,
// 786 -> 799 us; N = 36, 16 states 7.4e-7, 9.8e-7, 4.0e-7, 1.50 -> 1.52 ms (a part reads and writes the
// CTA's 64 KB of y).  Four parts gave 5.0e-7, 5.4e-7, 5.6e-7: their chunks hold unequal numbers of masks.
template <template <int, bool> class Arith, int RB, int SEC, bool LOWB, bool SHARE, int MAXT, int MINB, bool PARTS>
__global__ void __launch_bounds__(MAXT, MINB)
    k_apply_block(ApplyParams p, const BlockArgs c, const int4* __restrict__ chunks, const unsigned char* __restrict__ blob,
                  const void* __restrict__ psi, typename Arith<RB, SHARE>::Out* __restrict__ y) {
  using namespace blk;
  using A = Arith<RB, SHARE>;
  using Out = typename A::Out;
  using Sum = typename A::Sum;
  using Real = decltype(Out().x);
  constexpr int R = 1 << RB, kElem = A::kElem, kStages = A::kRing;
  const int SE = SEC ? SEC : c.SE;
  const int B = c.B, LB = c.LB, MB = c.MB;
  const int tileb = (SE << (RB + MB)) * kElem, stageb = tileb + c.auxb;
  extern __shared__ __align__(128) unsigned char sm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + kStages * stageb);
  int* done = reinterpret_cast<int*>(full + kStages);  // warps that finished the stage's chunk
  int* issued = done + kStages;                        // chunks copied into the stage so far
  int* lost = issued + kStages;                        // a wait gave up
  const int tid = threadIdx.x, nwarps = blockDim.x >> 5;
  const uint32_t crank = tma::cluster_rank(), csize = tma::cluster_size();  // 0 and 1 without clusters
  const uint32_t tile = blockIdx.x / csize;
  const int q0 = c.begin[crank], nq = c.begin[crank + 1] - q0;
  const bool active = tid < c.nt;
  const int t = active ? tid : 0;
  const int mid = t / SE, el = t - mid * SE, low = el / B, s = el - low * B;

  RowCtx ctx;
  ctx.x = (tile << (LB + RB + MB)) | ((uint32_t)mid << (LB + RB)) | (uint32_t)low;
  ctx.q = (uint32_t)(__popc(ctx.x) + p.sector) & 1u;
  ctx.above = (uint32_t)__popc(ctx.x >> (LB + RB)) & 1u;
  ctx.xn = (ctx.x & ((1u << LB) - 1u)) | ((ctx.x >> (LB + RB)) << LB);
  ctx.ng = (p.n - 1 - RB + 3) / 4;
  ctx.n = p.n;
  ctx.LB = LB;
  ctx.wd = static_cast<const float*>(p.wd);
  ctx.B = (uint32_t)B;
  ctx.share = reinterpret_cast<float2*>(sm + kStages * stageb + 64 + (SHARE ? (tid >> 5) * A::share(B) : 0));

  typename A::Acc acc;
  A::zero(acc);

  if (tid == 0) {
    for (int k = 0; k < kStages; ++k) {
      tma::mbar_init(&full[k], 1);
      done[k] = issued[k] = 0;
    }
    *lost = 0;
    tma::fence_mbar_init();
  }
  __syncthreads();
  auto issue = [&](int q, const int4 ch) {  // one thread
    const int st = q % kStages;
    ++issued[st];
    unsigned char* buf = sm + st * stageb;
    const uint32_t part = tile ^ ((uint32_t)ch.x & 0x7fffffffu);
    tma::expect_tx(&full[st], (uint32_t)tileb + (uint32_t)ch.z * 16u);
    tma::bulk_load(buf, reinterpret_cast<const unsigned char*>(psi) + (size_t)part * tileb, (uint32_t)tileb, &full[st]);
    tma::bulk_load(buf + tileb, blob + (size_t)ch.y * 16, (uint32_t)ch.z * 16u, &full[st]);
  };
  if (tid == 0)
    for (int q = 0; q < kStages && q < nq; ++q) issue(q, __ldg(&chunks[q0 + q]));

  int q = 0;
  for (int qe = PARTS ? min(c.part, nq) : nq;; qe = min(qe + c.part, nq)) {
    for (; q < qe; ++q) {
      const int st = q % kStages;
      // the refill's chunk is read ahead: the refill itself then starts at once
      const int4 refill = q + kStages < nq ? __ldg(&chunks[q0 + q + kStages]) : make_int4(0, 0, 0, 0);
      // the lanes of a warp go on or give up together: a lane that left the loop alone would keep the
      // others from ever passing the warp barriers below
      if (!__all_sync(0xffffffffu, tma::wait_bounded(&full[st], (q / kStages) & 1, tma::wait_polls()))) break;
      const unsigned char* tb = sm + st * stageb;
      const unsigned char* cb = tb + tileb;
      const uint4 head = *reinterpret_cast<const uint4*>(cb);
      const uint4* rec = reinterpret_cast<const uint4*>(cb) + 1;
      constexpr bool LOWS = SEC != 16 || LOWB;
      auto partner = [&](const uint4 rc) SYK_INLINE {  // the thread's partner row 0
        const uint32_t lm = LOWS ? (rc.x >> 16) & 0xffu : 0u;
        return tb + (size_t)((((uint32_t)mid ^ (rc.x & 0xffffu)) << RB) * SE + ((uint32_t)low ^ lm) * B + s) * kElem;
      };
      CosetAt next;
      uint4 rc;
      auto prepare = [&]() SYK_INLINE {  // the next record's coset
        rc = *rec++;
        next.odd = rc.x >> 31;
        next.prow = partner(rc);
        next.un = support(ctx.x, rc.z);
        next.sg = parity(rc.y & ctx.x);
        next.tb = cb + rc.w;
      };
      const uint32_t cn = head.x;
      auto run = [&](auto w, uint32_t count) SYK_INLINE {
        constexpr int W = decltype(w)::value;
  #pragma unroll 1
        for (uint32_t k = 0; k < count; ++k) {
          const CosetAt at = next;
          prepare();
          A::template coset<W, LOWS>(acc, at, SE * kElem, ctx, p);
          if (W == 4 && (k & 7u) == 7u) A::renorm(acc);
        }
        if (W == 4) A::renorm(acc);
      };
      prepare();  // (a record past the last one is never used: it reads the tables behind it)
      run(std::integral_constant<int, 4>{}, cn & 0xffu);
      run(std::integral_constant<int, 3>{}, (cn >> 8) & 0xffu);
      run(std::integral_constant<int, 2>{}, (cn >> 16) & 0xffu);
      run(std::integral_constant<int, 1>{}, cn >> 24);
      run(std::integral_constant<int, 0>{}, head.y & 0xffu);
  #pragma unroll 1
      for (uint32_t k = head.y >> 8; k > 0; --k) {
        const uint4 r2 = rc;
        rc = *rec++;
        A::record(acc, partner(r2), SE * kElem, r2, cb + r2.w, ctx);
      }
      // the warp that finishes the chunk last refills its stage
      __syncwarp();
      if ((tid & 31) == 0) {
        __threadfence_block();
        if (atomicAdd(&done[st], 1) == nwarps - 1) {
          __threadfence_block();  // the other warps' reads come before the refill's writes
          done[st] = 0;
          if (q + kStages < nq) issue(q + kStages, refill);
        }
      }
      __syncwarp();
    }
    if (!PARTS || q < qe || q == nq) break;  // (q < qe: a wait gave up)
    if constexpr (PARTS) {  // (a thread's rows of y are its own)
      if (active) {
        Out* __restrict__ yt = y + (size_t)tile * (tileb / kElem) + (size_t)(mid << RB) * SE + el;
        const bool first = q == c.part;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          Sum v = A::get(acc, r);
          if (!first) A::add(v, yt[r * SE]);
          yt[r * SE] = v;
        }
      }
      A::zero(acc);
    }
  }
  if (q < nq) *lost = 1;
  __syncthreads();
  if (*lost) {
    // let every copy still in flight land before the buffers are reused or the CTA exits
    if (tid == 0) {
      atomicOr(p.status, 4);
      for (int k = 0; k < kStages; ++k)
        if (issued[k]) tma::wait_bounded(&full[k], (issued[k] - 1) & 1, tma::kDrainPolls);
    }
    __syncthreads();
  }

  // outputs; the CTAs of a cluster add their sums through shared memory
  const Real sc = p.ep_part && p.ep_scale ? (Real)p.ep_scale[s] : Real(1);
  const size_t gbase = (size_t)tile * (tileb / kElem);
  double dr = 0.0, di = 0.0;
  Real fr = 0, fi = 0;  // flushed to FP64 every 16 elements
  const Out* __restrict__ u = static_cast<const Out*>(p.ep_u);
  // element e of the tile; k counts the thread's elements
  auto emit = [&](size_t e, Out v, int k) {
    if (p.ep_part) {
      v.x *= sc;
      v.y *= sc;
      const Out w = u[gbase + e];
      fr = fma(w.x, v.x, fma(w.y, v.y, fr));
      fi = fma(w.x, v.y, fma(-w.y, v.x, fi));
      if ((k & 15) == 15) {
        dr += fr;
        di += fi;
        fr = fi = 0;
      }
    }
    y[gbase + e] = v;
  };
  if (csize > 1) {
    Sum* st = reinterpret_cast<Sum*>(sm);
    if (active) {
#pragma unroll
      for (int r = 0; r < R; ++r) st[((mid << RB) + r) * SE + el] = A::get(acc, r);
    }
    tma::cluster_sync();
    // each CTA adds 1/csize of the tile's elements over the cluster, in rank order
    const int part = (tileb / kElem) / (int)csize;
    if (active) {
      int k = 0;
      for (int e = (int)crank * part + tid; e < ((int)crank + 1) * part; e += c.nt, ++k) {
        const uint32_t a = tma::saddr(st + e);
        Sum v = ld_cluster_elem<Sum>(tma::map_rank(a, 0));
        for (uint32_t r = 1; r < csize; ++r) A::add(v, ld_cluster_elem<Sum>(tma::map_rank(a, r)));
        emit((size_t)e, v, k);
      }
    }
    tma::cluster_sync();  // no CTA leaves, or reuses its memory, while others read it
  } else {
    if (active) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const size_t e = (size_t)((mid << RB) + r) * SE + el;
        Sum v = A::get(acc, r);
        if (PARTS && nq > c.part) A::add(v, y[gbase + e]);
        emit(e, v, r);
      }
    }
    __syncthreads();
  }
  if (p.ep_part) {
    // the CTA's sums per state: thread g * B + s holds state s of group g; halve the groups
    double2* red = reinterpret_cast<double2*>(sm);
    if (active) red[tid] = make_double2(dr + fr, di + fi);
    __syncthreads();
    for (int h = c.nt / B / 2; h > 0; h >>= 1) {
      if (tid < h * B) {
        red[tid].x += red[tid + h * B].x;
        red[tid].y += red[tid + h * B].y;
      }
      __syncthreads();
    }
    if (tid < B) p.ep_part[(size_t)blockIdx.x * B + tid] = red[tid];
    if (blockIdx.x == 0 && tid == 0) *p.ep_nblk = (int)gridDim.x;
  }
}

// The instantiations are spread over translation units (each takes a while to compile); which:
// the state counts they serve.
enum { kBlock16 = 0, kBlockShare = 1, kBlockPow2 = 2, kBlockAny = 3 };
int launch_block32_share(const ApplyParams& p, const BlockArgs& a, int which, int cs, const BlockLayout* L,
                         const void* psi, void* y, cudaStream_t st);
int launch_block32_parts(const ApplyParams& p, const BlockArgs& a, int which, const BlockLayout* L, const void* psi, void* y,
                         cudaStream_t st);
int launch_block_df(const ApplyParams& p, const BlockArgs& a, int cs, const BlockLayout* L, const void* psi, void* y,
                    cudaStream_t st);
int launch_block32_direct(const ApplyParams& p, const BlockArgs& a, int which, int cs, const BlockLayout* L,
                          const void* psi, void* y, cudaStream_t st);

template <template <int, bool> class Arith, int RB, int SEC, bool LOWB, bool SHARE, int MAXT, int MINB, bool PARTS = false>
int launch_block(const ApplyParams& p, const BlockArgs& a, int cs, const BlockLayout* L, const void* psi, void* y,
             cudaStream_t st) {
  const int tb = a.LB + RB + a.MB;
  const int64_t ntiles = p.D >> tb;
  if (p.ep_part && ntiles * cs > p.ep_cap) {
    set_error("apply_H: %lld CTAs exceed the epilogue buffer (%lld)", (long long)(ntiles * cs), (long long)p.ep_cap);
    return SYK_EINVAL;
  }
  using Out = typename Arith<RB, SHARE>::Out;
  const size_t smem = block_smem(a.B, a.LB, RB, a.MB, a.auxb, Arith<RB, SHARE>::kElem);
  const auto kern = k_apply_block<Arith, RB, SEC, LOWB, SHARE, MAXT, MINB, PARTS>;
  SYK_TRY(ensure_smem_limit((const void*)kern, (int)kMaxSmemPerCta));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(ntiles * cs), 1, 1);
  cfg.blockDim = dim3((unsigned)((a.nt + 31) / 32 * 32), 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cs > 1 ? 1 : 0;
  SYK_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kern, p, a, (const int4*)L->chunks, (const unsigned char*)L->blob,
                                    psi, static_cast<Out*>(y)));
  count_launch();
  count_matvec(Arith<RB, SHARE>::kElem == 8 ? kMvCoset : kMvTiled);
  SYK_CUDA_CHECK(cudaGetLastError());
  return SYK_OK;
}

}  // namespace syk
