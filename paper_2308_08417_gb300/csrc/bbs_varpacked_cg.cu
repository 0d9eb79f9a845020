// Uneven batches, CG with Jacobi: packed small-system kernels with 16 lanes per
// system, R = 1..kMaxPackedR rows per lane.
#include "bbs_varpacked.cuh"

namespace bbs {
static_assert(kMaxPackedR == 10, "the table covers R = 1..10");
const void* varpacked_fn_cg(int R) {
    static const void* const kTable[kMaxPackedR] = {
        (const void*)varpacked_kernel<1, true, 16, 1>, (const void*)varpacked_kernel<1, true, 16, 2>,
        (const void*)varpacked_kernel<1, true, 16, 3>, (const void*)varpacked_kernel<1, true, 16, 4>,
        (const void*)varpacked_kernel<1, true, 16, 5>, (const void*)varpacked_kernel<1, true, 16, 6>,
        (const void*)varpacked_kernel<1, true, 16, 7>, (const void*)varpacked_kernel<1, true, 16, 8>,
        (const void*)varpacked_kernel<1, true, 16, 9>, (const void*)varpacked_kernel<1, true, 16, 10>};
    return kTable[R - 1];
}
}  // namespace bbs
