// The CG scalars formed on the device by the last block of the pass that sums them (cg.cu, sym_tc.cu).
#pragma once

#include "internal.cuh"

namespace krr {

// True in every thread of the grid's last block to get here: the blocks' global writes before the
// call are then visible to it.  *ticket starts at 0 and is 0 again afterwards.
__device__ __forceinline__ bool last_block(unsigned* ticket) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(ticket, 1u) == gridDim.x * gridDim.y - 1;
        if (last) *ticket = 0;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// sum of column q's per-block partials, in every lane (read past L1: another block of the same launch
// may have written them)
__device__ __forceinline__ double warp_sum_parts(const double* __restrict__ part, int nblk, int q) {
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    for (int b = lane; b < nblk; b += 32) s += __ldcg(part + (size_t)q * nblk + b);
    return warp_sum(s);
}

// a_q = rz_q / (p_q . q_q) for active columns; zero otherwise (one warp; s = p_q . q_q).
__device__ __forceinline__ void cg_alpha(CGScalars* cg, int q, double s) {
    cg->pq[q] = s;
    double a = 0.0;
    if (cg->active[q]) {
        if (!(s > 0.0) || !isfinite(s) || !isfinite(cg->rz[q])) {
            cg->bad = 1;
            cg->active[q] = 0;
        } else {
            a = cg->rz[q] / s;
        }
    }
    cg->a[q] = a;
}

}  // namespace krr
