// Reductions of several values at once and 16-byte element access, shared by
// the vector kernels.
#pragma once

#include "dwf_internal.cuh"

namespace dwf {

namespace {

// 16 bytes of a field: two FP32 elements or one FP64 element
template <typename T> struct Pack;
template <> struct Pack<float2> {
    static constexpr int N = 2;
    float2 e[2];
};
template <> struct Pack<double2> {
    static constexpr int N = 1;
    double2 e[1];
};
template <typename T> __device__ __forceinline__ Pack<T> ldp(const T *p, int64_t i) {  // packs i
    Pack<T> r;
    *reinterpret_cast<float4 *>(&r) = reinterpret_cast<const float4 *>(p)[i];
    return r;
}
template <typename T> __device__ __forceinline__ void stp(T *p, int64_t i, const Pack<T> &v) {
    reinterpret_cast<float4 *>(p)[i] = *reinterpret_cast<const float4 *>(&v);
}

__host__ __device__ constexpr int pow2_at_least(int n) { return n <= 1 ? 1 : 2 * pow2_at_least((n + 1) / 2); }
__host__ __device__ constexpr int log2_of(int n) { return n <= 1 ? 0 : 1 + log2_of(n / 2); }

// Sum of each of N (a power of two, at most 32) values over the warp: every
// step a lane keeps one half of the values it holds and adds the partner's
// share of them, N - 1 + log2(32 / N) additions where one value at a time takes
// 5 N (FP64 additions are this chip's slowest: 16 cycles of an SM per warp).
// Lane l returns the sum of value l >> (5 - log2 N).
template <int N> __device__ __forceinline__ double warp_sums(double (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int n = N; n > 1; n >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < N / 2; ++i)
            if (i < n / 2) {
                const double send = up ? v[i] : v[i + n / 2], keep = up ? v[i + n / 2] : v[i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
    }
#pragma unroll
    for (int k = 0; k < 5 - log2_of(N); ++k, o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

// The M values v of every thread summed over the grid's blockIdx.x, in a fixed
// order: the last CTA (atomic ticket) adds the partials part[i * gridDim.x + cta]
// and writes value i to out[i], i < nout.
template <int M>
__device__ void grid_sums(const double (&mine)[M], double *part, unsigned *count, double *out, int nout) {
    constexpr int N = pow2_at_least(M);
    __shared__ double sh[32][N];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5, nb = gridDim.x;
    double v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = i < M ? mine[i] : 0.0;
    const double t = warp_sums<N>(v);
    if ((lane & (32 / N - 1)) == 0) sh[warp][lane >> (5 - log2_of(N))] = t;
    __syncthreads();
    if (threadIdx.x < M) {
        double u = 0;
        for (int w = 0; w < nw; ++w) u += sh[w][threadIdx.x];
        part[(size_t)threadIdx.x * nb + blockIdx.x] = u;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(count, 1u) == (unsigned)nb - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int i = warp; i < nout; i += nw) {
        double s = 0;
        for (int k = lane; k < nb; k += 32) s += __ldcg(part + (size_t)i * nb + k);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) out[i] = s;
    }
    if (threadIdx.x == 0) *count = 0u;
}

}  // namespace

}  // namespace dwf
