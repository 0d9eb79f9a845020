// Uneven batches, one block per system: BiCGSTAB with Jacobi on staged values
// (block fixed point, or FP64 where a system does not fit it), for the systems
// above the packed sizes.
//
// The planner groups the systems by (warps, rows per thread), as the uniform
// batches are launched: the fewest warps, a power of two, that leave at most 8
// rows a thread. Each group is a launch of varteam_kernel<R> in the plan's graph.
// Team systems run in persistent launches: as many blocks as stay resident, each
// taking the group's next system from a counter. Wide teams (bbs_var_tuning.wide)
// have a block for each system.
//
// Against one persistent kernel of 8-warp blocks that holds every team size and
// every rows-per-thread variant (bbs_varsize.cuh, which still runs CG and
// unpreconditioned systems and those too large to stage): that kernel takes 255
// registers for its largest variant, 8 warps an SM, and its warps run different
// variants side by side, whose code evicts each other's from the instruction
// cache. 20,000 systems, n log-uniform in 16..1024: 13.04 ms with
// that kernel, 6.40 ms with these.
#pragma once

#include <cstdint>

#include "bbs_fixed.cuh"

namespace bbs {

struct VarTeamParams {
    const int32_t* pat_n;
    const int32_t* pat_nnz;
    const int64_t* rp_off;
    const int64_t* ci_off;
    const int32_t* row_ptrs;
    const int32_t* col_idxs;
    const int32_t* sys_pattern;
    const int64_t* val_off;
    const int64_t* vec_off;
    const double* values;
    const double* b;
    double* x;
    int32_t* iters;
    double* rel_res;
    int32_t* status;
    const int32_t* order;  // the group's systems
    int32_t* counter;      // the next system to take, or null: one block for each
    int count;
    SolveCfg cfg;
};

// Block area: item (16 bytes) | red [256 doubles] | xa [n_pad] | xb [n_pad] | staged values.
template <int R>
__global__ void __launch_bounds__(256, 1) varteam_kernel(const __grid_constant__ VarTeamParams P) {
    extern __shared__ __align__(16) unsigned char raw[];
    const Team tm = Team::block();
    int* cell = reinterpret_cast<int*>(raw);
    for (int item = blockIdx.x;;) {
        if (P.counter != nullptr) {
            if (tm.tid == 0) *cell = atomicAdd(P.counter, 1);
            __syncthreads();
            item = *cell;
        }
        if (item >= P.count) break;
        const int sys = ldg(P.order + item);
        const int pat = ldg(P.sys_pattern + sys);
        const int n = ldg(P.pat_n + pat);
        const Mat<double> A{P.values + ldg(P.val_off + sys), P.row_ptrs + ldg(P.rp_off + pat),
                            P.col_idxs + ldg(P.ci_off + pat), n, 0};
        const int64_t vo = ldg(P.vec_off + sys);
        SysIO io;
        io.b = P.b + vo;
        io.x = P.x + vo;
        io.iters = P.iters + sys;
        io.rel_res = P.rel_res + sys;
        io.status = P.status + sys;
        io.inner = nullptr;
        io.n = n;
        const TeamSmem sm = team_smem(raw + 16, (n + 1) & ~1);
        const size_t nnz = (size_t)ldg(P.pat_nnz + pat);
        const auto op = make_op<FMT_CSR, R>(A, nnz, sm.extra, tm);
        bicgstab_staged_jacobi<FMT_CSR, R>(op, nnz, io, P.cfg, sm, tm);
        if (P.counter == nullptr) break;
        __syncthreads();  // every thread has read its item and is done with the area
    }
}

// Shared-memory bytes of a block for a system of n rows and nnz values.
__host__ __device__ constexpr size_t varteam_smem(int n, int nnz) {
    return 16 + (256 + 2 * (size_t)((n + 1) & ~1)) * 8 + (((size_t)nnz * 8 + 15) & ~(size_t)15);
}

// Kernel of R rows per thread (1..kMaxR).
const void* varteam_fn(int R);
const void* varteam_fn_lo(int R);
const void* varteam_fn_hi(int R);

}  // namespace bbs
