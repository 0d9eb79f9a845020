// Packed BiCGSTAB, CG and GMRES kernels (32 / L systems per warp) without a
// preconditioner, CSR format, L = 4 lanes per system, R = 1..kMaxPackedR rows per lane.
#include "bbs_kernels.h"
#include "bbs_packed.cuh"

namespace bbs {
#define BBS_TABLE(K) \
    static const void* const kTable[kMaxPackedR] = { \
        (const void*)K<FMT_CSR, 4, 1>, (const void*)K<FMT_CSR, 4, 2>, \
        (const void*)K<FMT_CSR, 4, 3>, (const void*)K<FMT_CSR, 4, 4>, \
        (const void*)K<FMT_CSR, 4, 5>, (const void*)K<FMT_CSR, 4, 6>, \
        (const void*)K<FMT_CSR, 4, 7>, (const void*)K<FMT_CSR, 4, 8>, \
        (const void*)K<FMT_CSR, 4, 9>, (const void*)K<FMT_CSR, 4, 10>}; \
    return kTable[R - 1];
static_assert(kMaxPackedR == 10, "tables cover R = 1..10");
const void* bicgstab_plain_packed_fn_csr_l4(int R) { BBS_TABLE(bicgstab_plain_packed_kernel) }
const void* gmres_plain_packed_fn_csr_l4(int R) { BBS_TABLE(gmres_plain_packed_kernel) }
const void* cg_plain_packed_fn_csr_l4(int R) { BBS_TABLE(cg_plain_packed_kernel) }
#undef BBS_TABLE
}  // namespace bbs
