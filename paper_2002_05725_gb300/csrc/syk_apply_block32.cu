// Row-block matvec with 32 rows per thread for 1, 2 and 4 states and for state counts that are no
// power of two (see syk_block_kernel.cuh).
#include "syk_block_kernel.cuh"

namespace syk {

int launch_block32_direct(const ApplyParams& p, const BlockArgs& a, int which, int cs, const BlockLayout* L,
                          const void* psi, void* y, cudaStream_t st) {
  return which == kBlockPow2 ? launch_block<BlockF32, 5, 16, true, false, 256, 1>(p, a, cs, L, psi, y, st)
                             : launch_block<BlockF32, 5, 0, true, false, 256, 1>(p, a, cs, L, psi, y, st);
}

}  // namespace syk
