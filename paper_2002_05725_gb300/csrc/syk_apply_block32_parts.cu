// Row-block matvec with 32 rows per thread for 8 and 16 states whose sums are taken in parts (see
// syk_block_kernel.cuh).
#include "syk_block_kernel.cuh"

namespace syk {

int launch_block32_parts(const ApplyParams& p, const BlockArgs& a, int which, const BlockLayout* L, const void* psi, void* y,
                         cudaStream_t st) {
  return which == kBlock16 ? launch_block<BlockF32, 5, 16, false, true, 256, 1, true>(p, a, 1, L, psi, y, st)
                           : launch_block<BlockF32, 5, 16, true, true, 256, 1, true>(p, a, 1, L, psi, y, st);
}

}  // namespace syk
