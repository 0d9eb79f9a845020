// Uneven batches: one-block-per-system kernels with 6 to 8 rows per thread.
#include "bbs_varteam.cuh"

namespace bbs {
const void* varteam_fn_hi(int R) {
    static const void* const kTable[3] = {(const void*)varteam_kernel<6>, (const void*)varteam_kernel<7>,
                                          (const void*)varteam_kernel<8>};
    return kTable[R - 6];
}
static_assert(kMaxR == 8, "tables cover R = 1..8");
}  // namespace bbs
