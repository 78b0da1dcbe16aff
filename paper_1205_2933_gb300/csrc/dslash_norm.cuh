// The output norms that the Dslash kernels sum in their epilogues.
#pragma once

#include "dwf_internal.cuh"

namespace dwf {

namespace {

// Where a right-hand side's |out|^2 goes: one FP64 partial per CTA, added in a
// fixed order into slot[r * stride].  With `count` (a zeroed counter per
// right-hand side) the last CTA to finish adds them; else norm_finish_kernel
// does.  The counter saves a launch, but the CTAs' atomics on one address take
// their turns: 120 CTAs (8x6x4x10x8) gain 2 us per Dslash, 1024 lose 4 us.
struct NormOut {
    double *part;     // [nrhs][gridDim.x]
    double *slot;
    unsigned *count;
    int stride;
};

// v: the warp's share of |out_r|^2, in lane 0; every thread of the CTA calls it.  sh: 33 doubles
__device__ __forceinline__ void norm_epilogue(const NormOut &n, int r, double v, double *sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int w = 0; w < nw; ++w) t += sh[w];
        n.part[(size_t)r * gridDim.x + blockIdx.x] = t;
        if (n.count) {
            __threadfence();
            sh[32] = atomicAdd(n.count + r, 1u) == gridDim.x - 1 ? 1.0 : 0.0;
        }
    }
    __syncthreads();  // (sh is also rewritten for the next right-hand side)
    if (!n.count) return;
    if (sh[32] != 0.0) {
        __threadfence();
        double t = 0;
        for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) t += __ldcg(n.part + (size_t)r * gridDim.x + i);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if (lane == 0) sh[warp] = t;
        __syncthreads();
        if (threadIdx.x == 0) {
            double u = 0;
            for (int w = 0; w < nw; ++w) u += sh[w];
            n.slot[(size_t)r * n.stride] = u;
            n.count[r] = 0u;
        }
    }
    __syncthreads();
}

// nslot[r * nstride] = sum of the nb CTA partials of right-hand side r = blockIdx.x (fixed order)
__global__ void __launch_bounds__(1024) norm_finish_kernel(const double *npart, double *nslot,
                                                           int nstride, int nb) {
    __shared__ double red[32];
    pdl_wait();
    pdl_dependents();
    const double *pr = npart + (size_t)blockIdx.x * nb;
    double t = 0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) t += pr[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double u = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) u += red[w];
        nslot[(size_t)blockIdx.x * nstride] = u;
    }
}

// partials for `grid` and, up to 256 CTAs per right-hand side, the counters
NormOut norm_out(dwf_ctx *c, dim3 grid, int nrhs, double *slot, int stride) {
    const size_t pb = sizeof(double) * (size_t)grid.x * nrhs;
    if (c->dn_part.bytes < pb) c->dn_part.alloc(pb);
    const bool few = grid.x <= 256 && nrhs <= DN_COUNTERS;
    return NormOut{c->dn_part.as<double>(), slot, few ? c->dn_count.as<unsigned>() : nullptr, stride};
}

void norm_finish(dwf_ctx *c, const NormOut &n, dim3 grid, int nrhs) {
    if (n.count) return;
    launch_after(norm_finish_kernel, dim3(nrhs), dim3(1024), 0, c->stream, n.part, n.slot, n.stride, (int)grid.x);
    DWF_CHECK_LAUNCH();
}

}  // namespace

}  // namespace dwf
