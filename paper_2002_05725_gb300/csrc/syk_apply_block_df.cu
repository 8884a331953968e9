// Row-block complex128 matvec in double-float arithmetic with 8 rows per thread, for 1, 2 and 4
// states (see syk_block_kernel.cuh, syk_block_df.cuh).
#include "syk_block_kernel.cuh"

namespace syk {

int launch_block_df(const ApplyParams& p, const BlockArgs& a, int cs, const BlockLayout* L, const void* psi, void* y,
                    cudaStream_t st) {
  return launch_block<BlockDf, 3, 16, true, false, 256, 2>(p, a, cs, L, psi, y, st);
}

}  // namespace syk
