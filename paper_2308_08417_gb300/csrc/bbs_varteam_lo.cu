// Uneven batches: one-block-per-system kernels with 1 to 5 rows per thread.
#include "bbs_varteam.cuh"

namespace bbs {
const void* varteam_fn_lo(int R) {
    static const void* const kTable[5] = {(const void*)varteam_kernel<1>, (const void*)varteam_kernel<2>,
                                          (const void*)varteam_kernel<3>, (const void*)varteam_kernel<4>,
                                          (const void*)varteam_kernel<5>};
    return kTable[R - 1];
}
}  // namespace bbs
