// Kernel of the fused coarsest-level GCR (one cooperative launch), shared by
// the 9-point (R D P) and 33-point (P^+ D^+ D P) stencils; each includer
// instantiates one stencil size.
#pragma once

#include <cooperative_groups.h>

#include "mg.cuh"

namespace dwf {

namespace cg = cooperative_groups;

namespace {

constexpr int CT = 256;        // threads per CTA
constexpr int MAXR = 32;       // maximum restart length of the fused solver

template <typename LT> struct LRead;
template <> struct LRead<double2> {
    template <typename R> static __device__ __forceinline__ C<R> get(const double2 *Y, int64_t i) { return cvt<C<R>, double2>(Y[i]); }
};
template <> struct LRead<float2> {
    template <typename R> static __device__ __forceinline__ C<R> get(const float2 *Y, int64_t i) { return cvt<C<R>, float2>(Y[i]); }
};
template <> struct LRead<__nv_bfloat162> {
    template <typename R> static __device__ __forceinline__ C<R> get(const __nv_bfloat162 *Y, int64_t i) {
        return cvt<C<R>, float2>(__bfloat1622float2(Y[i]));
    }
};
template <> struct LRead<__half2> {
    template <typename R> static __device__ __forceinline__ C<R> get(const __half2 *Y, int64_t i) {
        return cvt<C<R>, float2>(__half22float2(Y[i]));
    }
};

template <typename R, typename LT> struct Args {
    const LT *Y;
    const int *nbr;    // neighbour table [V][NPTS - 1]
    Geom g;            // coarse lattice (g.V sites)
    const C<R> *b;
    C<R> *x, *r, *Z, *W;   // Z, W: restart vectors each
    double2 *part;     // [3][MAXR + 2][gridDim.x] FP64 partial sums
    double tol;
    int maxiter, restart;
    int *iters;        // accumulates the iteration count
};

// out = A in on the owned sites [s0, s1): one warp per site, lane l holds
// column l of every link row (coalesced loads) and the 9 neighbour values
// in[nbr_d][l]; each output row is a warp-wide sum over l.
template <typename R, typename LT, int NV, int NPTS>
__device__ void apply_owned(const Args<R, LT> &a, C<R> *out, const C<R> *in, int64_t s0, int64_t s1) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool on = lane < NV;
    for (int64_t site = s0 + warp; site < s1; site += CT / 32) {
        C<R> xv[NPTS];
#pragma unroll
        for (int d = 0; d < NPTS; ++d) {
            const int o = d > 0 ? a.nbr[site * (NPTS - 1) + d - 1] : (int)site;
            xv[d] = on ? in[o * NV + lane] : mk<R>(0, 0);
        }
        const LT *Ys = a.Y + site * NPTS * NV * NV;
        // unrolled so that the link loads of several row pairs are in flight
        // together (the loop is bound by L2 latency, not bandwidth)
#pragma unroll 4
        for (int k = 0; k < NV; k += 2) {
            R r0 = 0, i0 = 0, r1 = 0, i1 = 0;
            if (on) {
#pragma unroll
                for (int d = 0; d < NPTS; ++d) {
                    C<R> y0 = LRead<LT>::template get<R>(Ys, ((int64_t)d * NV + k) * NV + lane);
                    C<R> y1 = LRead<LT>::template get<R>(Ys, ((int64_t)d * NV + k + 1) * NV + lane);
                    r0 += y0.x * xv[d].x - y0.y * xv[d].y;
                    i0 += y0.x * xv[d].y + y0.y * xv[d].x;
                    r1 += y1.x * xv[d].x - y1.y * xv[d].y;
                    i1 += y1.x * xv[d].y + y1.y * xv[d].x;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                r0 += __shfl_xor_sync(0xffffffffu, r0, o);
                i0 += __shfl_xor_sync(0xffffffffu, i0, o);
                r1 += __shfl_xor_sync(0xffffffffu, r1, o);
                i1 += __shfl_xor_sync(0xffffffffu, i1, o);
            }
            if (lane == 0) {
                out[site * NV + k] = mk<R>(r0, i0);
                out[site * NV + k + 1] = mk<R>(r1, i1);
            }
        }
    }
    // rows were written by lane 0 of each warp; the element loops that follow
    // read them from other threads of the CTA
    __syncthreads();
}

// Sum over CTAs of part[slot][i][*] for i < k into tot[i] (shared), same
// order in every CTA.  16 lanes per value.
__device__ void gather_totals(const double2 *part, int k, int nb, double2 *tot) {
    for (int i0 = 0; i0 < k; i0 += CT / 16) {
        const int i = i0 + threadIdx.x / 16, lane = threadIdx.x & 15;
        double2 s = make_double2(0, 0);
        if (i < k)
            for (int b = lane; b < nb; b += 16) {
                const volatile double *p = reinterpret_cast<const volatile double *>(part + (size_t)i * nb + b);
                s.x += p[0];
                s.y += p[1];
            }
        for (int o = 8; o > 0; o >>= 1) {
            s.x += __shfl_down_sync(0xffffffffu, s.x, o, 16);
            s.y += __shfl_down_sync(0xffffffffu, s.y, o, 16);
        }
        if (i < k && lane == 0) tot[i] = s;
    }
    __syncthreads();
}

// The solver with its vectors in global memory: for directions that do not fit
// the SMs' shared memory (coarse_gcr_smem_kernel below takes the others).
template <typename R, typename LT, int NV, int NPTS>
__global__ void __launch_bounds__(CT) coarse_gcr_kernel(Args<R, LT> a) {
    cg::grid_group grid = cg::this_grid();
    __shared__ double2 red[CT / 32][MAXR + 2];
    __shared__ double2 tot[MAXR + 2];
    const int nb = gridDim.x;
    const int64_t N = a.g.V * NV;
    const int64_t sites = (a.g.V + nb - 1) / nb;   // whole sites per CTA
    const int64_t s0 = blockIdx.x * sites;
    const int64_t s1 = s0 + sites < a.g.V ? s0 + sites : a.g.V;
    const int64_t e0 = s0 * NV;
    const int64_t e1 = s1 > s0 ? s1 * NV : e0;
    const size_t ps = (size_t)(MAXR + 2) * nb;   // size of one partial-sum region
    double2 *P[3] = {a.part, a.part + ps, a.part + 2 * ps};

    // reduce k complex values per thread into tot[0..k): warp shuffles for
    // all k values, one shared-memory pass across warps, one partial per CTA
    auto reduce = [&](double2 *vals, int k, double2 *Pr) {
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        for (int i = 0; i < k; ++i) {
            double2 t = vals[i];
            for (int o = 16; o > 0; o >>= 1) {
                t.x += __shfl_down_sync(0xffffffffu, t.x, o);
                t.y += __shfl_down_sync(0xffffffffu, t.y, o);
            }
            if (lane == 0) red[w][i] = t;
        }
        __syncthreads();
        if (threadIdx.x < k) {
            double2 t = make_double2(0, 0);
            for (int j = 0; j < CT / 32; ++j) {
                t.x += red[j][threadIdx.x].x;
                t.y += red[j][threadIdx.x].y;
            }
            Pr[(size_t)threadIdx.x * nb + blockIdx.x] = t;
        }
        __threadfence();
        grid.sync();
        gather_totals(Pr, k, nb, tot);
    };

    // x = 0, r = b, |b|^2
    double2 v[MAXR + 2];
    v[0] = make_double2(0, 0);
    for (int64_t e = e0 + threadIdx.x; e < e1; e += CT) {
        a.x[e] = mk<R>(0, 0);
        C<R> bv = a.b[e];
        a.r[e] = bv;
        v[0].x += (double)bv.x * bv.x + (double)bv.y * bv.y;
    }
    reduce(v, 1, P[2]);
    const double bn2 = tot[0].x;
    double rn2 = bn2;
    int it = 0, k = 0;
    if (bn2 > 0.0) {
        const double stop = a.tol * a.tol * bn2;
        while (it < a.maxiter && rn2 > stop) {
            C<R> *Zk = a.Z + (size_t)k * N, *Wk = a.W + (size_t)k * N;
            for (int64_t e = e0 + threadIdx.x; e < e1; e += CT) Zk[e] = a.r[e];
            __threadfence();
            grid.sync();
            apply_owned<R, LT, NV, NPTS>(a, Wk, Zk, s0, s1);
            for (int pass = 0; pass < 2 && k > 0; ++pass) {
                for (int i = 0; i < k; ++i) v[i] = make_double2(0, 0);
                for (int64_t e = e0 + threadIdx.x; e < e1; e += CT) {
                    C<R> w = Wk[e];
                    // loads issued eight at a time before the products (the loop is latency-bound)
                    for (int i0 = 0; i0 < k; i0 += 8) {
                        C<R> u[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (i0 + j < k) u[j] = a.W[(size_t)(i0 + j) * N + e];
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (i0 + j < k) {
                                v[i0 + j].x += (double)u[j].x * w.x + (double)u[j].y * w.y;
                                v[i0 + j].y += (double)u[j].x * w.y - (double)u[j].y * w.x;
                            }
                    }
                }
                reduce(v, k, P[pass]);
                for (int64_t e = e0 + threadIdx.x; e < e1; e += CT) {
                    C<R> w = Wk[e], z = Zk[e];
                    for (int i0 = 0; i0 < k; i0 += 8) {
                        C<R> wi[8], zi[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (i0 + j < k) {
                                wi[j] = a.W[(size_t)(i0 + j) * N + e];
                                zi[j] = a.Z[(size_t)(i0 + j) * N + e];
                            }
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (i0 + j < k) {
                                const R br = (R)tot[i0 + j].x, bi = (R)tot[i0 + j].y;
                                w.x -= br * wi[j].x - bi * wi[j].y;
                                w.y -= br * wi[j].y + bi * wi[j].x;
                                z.x -= br * zi[j].x - bi * zi[j].y;
                                z.y -= br * zi[j].y + bi * zi[j].x;
                            }
                    }
                    Wk[e] = w;
                    Zk[e] = z;
                }
                __syncthreads();  // tot is rewritten by the next reduction
            }
            v[0] = v[1] = make_double2(0, 0);
            for (int64_t e = e0 + threadIdx.x; e < e1; e += CT) {
                C<R> w = Wk[e], rr = a.r[e];
                v[0].x += (double)w.x * w.x + (double)w.y * w.y;
                v[1].x += (double)w.x * rr.x + (double)w.y * rr.y;
                v[1].y += (double)w.x * rr.y - (double)w.y * rr.x;
            }
            reduce(v, 2, P[2]);
            const double ww = tot[0].x;
            if (!(ww > 0.0)) break;  // breakdown: same decision in every CTA
            const double inv = 1.0 / sqrt(ww);
            const double ar = tot[1].x * inv, ai = tot[1].y * inv;
            const R sc = (R)inv, arr = (R)ar, aii = (R)ai;
            for (int64_t e = e0 + threadIdx.x; e < e1; e += CT) {
                C<R> z = Zk[e], w = Wk[e], xx = a.x[e], rr = a.r[e];
                z.x *= sc; z.y *= sc; w.x *= sc; w.y *= sc;
                xx.x += arr * z.x - aii * z.y;
                xx.y += arr * z.y + aii * z.x;
                rr.x -= arr * w.x - aii * w.y;
                rr.y -= arr * w.y + aii * w.x;
                Zk[e] = z; Wk[e] = w; a.x[e] = xx; a.r[e] = rr;
            }
            rn2 -= ar * ar + ai * ai;
            ++it;
            ++k;
            __syncthreads();
            if (k == a.restart || rn2 <= stop) {
                // true residual r = b - A x
                __threadfence();
                grid.sync();
                apply_owned<R, LT, NV, NPTS>(a, a.r, a.x, s0, s1);
                v[0] = make_double2(0, 0);
                for (int64_t e = e0 + threadIdx.x; e < e1; e += CT) {
                    C<R> bv = a.b[e], ax = a.r[e];
                    C<R> rr = mk<R>(bv.x - ax.x, bv.y - ax.y);
                    a.r[e] = rr;
                    v[0].x += (double)rr.x * rr.x + (double)rr.y * rr.y;
                }
                reduce(v, 1, P[2]);
                rn2 = tot[0].x;
                k = 0;
                __syncthreads();
            }
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(a.iters, it);
}

// ---- the solver with its vectors in shared memory ---------------------------
//
// Sums that cross threads and CTAs: FP64 for FP64 fields (and |b|^2); for FP32 fields the
// unevaluated sum of two FP32 numbers (about 48 bits), because an FP64 addition
// takes this chip's SM as long as 64 FP32 ones and every CTA adds up all
// partials of a reduction.
struct FF {
    float hi, lo;
};
__device__ __forceinline__ void acc_init(FF &a) { a.hi = a.lo = 0.f; }
__device__ __forceinline__ void acc_init(double &a) { a = 0.0; }
__device__ __forceinline__ void acc_add(FF &a, FF b) {  // two-sum of the high parts
    const float t = a.hi + b.hi, q = t - a.hi;
    const float e = (a.hi - (t - q)) + (b.hi - q) + (a.lo + b.lo);
    a.hi = t + e;
    a.lo = e - (a.hi - t);
}
__device__ __forceinline__ void acc_add(double &a, double b) { a += b; }
__device__ __forceinline__ void acc_fma(FF &a, float x, float y) {  // a += x y, the product exact
    const float p = __fmul_rn(x, y);  // not contracted with the addition that follows
    acc_add(a, FF{p, fmaf(x, y, -p)});
}
__device__ __forceinline__ void acc_fma(double &a, double x, double y) { a += x * y; }
__device__ __forceinline__ FF acc_xor(FF a, int o) {
    return FF{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}
__device__ __forceinline__ double acc_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ double acc_value(FF a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ double acc_value(double a) { return a; }
template <typename R> struct AccT;
template <> struct AccT<float> { using type = FF; };
template <> struct AccT<double> { using type = double; };
template <typename A> struct alignas(16) AccC {  // a complex partial sum, one 16-byte access
    A re, im;
};

// sites per CTA and shared-memory layout of the solver for V sites on at most `ctas` CTAs
template <typename R, typename LT, int NV, int NPTS> struct SmemPlan {
    static constexpr int LROW0 = NV * (int)sizeof(LT);                       // a link row
    // an odd number of 16-byte units, so that the rows of 8 lanes lie in 8 bank groups
    static constexpr int LROW = LROW0 % 32 == 0 ? LROW0 + 16 : LROW0;
    int64_t spc;
    size_t vec, stage, links, total;
    bool cached;  // the links fit as well
    SmemPlan(int64_t V, int restart, int64_t ctas, size_t limit) {
        spc = (V + ctas - 1) / ctas;
        vec = ((size_t)spc * NV * sizeof(C<R>) + 15) / 16 * 16;
        stage = (size_t)spc * NPTS * NV * sizeof(C<R>);
        stage = (stage + 15) / 16 * 16;
        links = (size_t)spc * NPTS * NV * LROW;
        const size_t base = vec * (2 * (size_t)restart + 2) + 2 * stage;
        cached = base + links <= limit;
        total = base + (cached ? links : 0);
    }
};

// the sum of N values (a power of two) in pairs
template <int N, typename T> __device__ __forceinline__ T pair_sum(const T (&v)[N]) {
    T t[N];
#pragma unroll
    for (int i = 0; i < N; ++i) t[i] = v[i];
#pragma unroll
    for (int h = N / 2; h >= 1; h /= 2)
#pragma unroll
        for (int i = 0; i < h; ++i) t[i] = t[i] + t[i + h];
    return t[0];
}

template <typename R, typename LT, int NV> __device__ __forceinline__ C<R> row_times(const unsigned char *row, const C<R> *x) {
    // NV links of one row in accesses of 16 bytes (8 where the row is no multiple),
    // summed in several chains of at most four links: one chain of 24 rounds 1.4
    // times worse than the warp-wide sum of the kernel above
    constexpr int NA = NV % 8 == 0 ? 8 : NV % 4 == 0 ? 4 : 2;
    constexpr int B = NV * sizeof(LT) % 16 == 0 ? 16 : 8;
    constexpr int E = B / (int)sizeof(LT) > 0 ? B / (int)sizeof(LT) : 1;
    struct alignas(B) Chunk {
        LT e[E];
    };
    C<R> acc[NA];
#pragma unroll
    for (int i = 0; i < NA; ++i) acc[i] = mk<R>(0, 0);
    constexpr int NCH = NV / E;
    Chunk ch[NCH < 8 ? NCH : 8];
#pragma unroll
    for (int c0 = 0; c0 < NCH; c0 += 8) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (c0 + i < NCH) ch[i] = *reinterpret_cast<const Chunk *>(row + (size_t)(c0 + i) * sizeof(Chunk));
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (c0 + i < NCH)
#pragma unroll
                for (int j = 0; j < E; ++j)
                    cfma(acc[((c0 + i) * E + j) % NA], LRead<LT>::template get<R>(ch[i].e, j), x[(c0 + i) * E + j]);
    }
    return pair_sum<NA>(acc);
}

// The same GCR, with what a CTA owns of every vector (the directions Z and W,
// x, r) and, where they fit, its sites' links in shared memory: only the
// vector the stencil acts on crosses CTAs, through a.r, and each iteration
// leaves the chip's SMs twice: one grid barrier to publish that vector, one
// for the reduction.  The products <W_i, w>, |w|^2 and <w, r> are reduced
// together: with W orthonormal |w|^2 loses sum |<W_i, w>|^2 in the projection
// and <w, r> does not change (r is orthogonal to the W_i).  Where the
// projection took a tenth or more of |w|^2, where that difference and the W_i's
// rounding would lose digits, a second one follows with a reduction of its own
// (at 3/4 FP64 rounds 1.1 times worse than with two projections each, at a
// hundredth no better).  The stencil: one
// thread per (direction, row) of a site, the neighbours' values staged.
// Bound by the latency of the two barriers and of one L2 round trip after
// each: 512 sites x 24 in BF16 52 us a call where the vectors in global memory,
// four barriers per iteration and FP64 sums took 117; 256 sites x 16 in FP64 (a
// V-cycle's) 0.09 ms against 0.67.
template <typename R, typename LT, int NV, int NPTS>
__global__ void __launch_bounds__(CT) coarse_gcr_smem_kernel(Args<R, LT> a, int spc, int cached) {
    using A = typename AccT<R>::type;
    using P = SmemPlan<R, LT, NV, NPTS>;
    cg::grid_group grid = cg::this_grid();
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ double2 tot[MAXR + 2];
    const int nb = gridDim.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int s0 = blockIdx.x * spc, ns = max(0, min(spc, (int)a.g.V - s0)), own = ns * NV;
    const int64_t e0 = (int64_t)s0 * NV;
    const size_t vec = ((size_t)spc * NV * sizeof(C<R>) + 15) / 16 * 16;
    const size_t stage = ((size_t)spc * NPTS * NV * sizeof(C<R>) + 15) / 16 * 16;
    auto W = [&](int i) { return reinterpret_cast<C<R> *>(sm + vec * i); };
    auto Z = [&](int i) { return reinterpret_cast<C<R> *>(sm + vec * (a.restart + i)); };
    C<R> *x = reinterpret_cast<C<R> *>(sm + vec * 2 * a.restart), *r = reinterpret_cast<C<R> *>(sm + vec * (2 * a.restart + 1));
    C<R> *sin = reinterpret_cast<C<R> *>(sm + vec * (2 * a.restart + 2));
    C<R> *sp = reinterpret_cast<C<R> *>(sm + vec * (2 * a.restart + 2) + stage);
    unsigned char *sl = sm + vec * (2 * a.restart + 2) + 2 * stage;
    C<R> *pub = a.r;  // the published vector

    if (cached) {
        constexpr int WR = P::LROW0 / 4;  // 4-byte words of a link row
        const unsigned *src = reinterpret_cast<const unsigned *>(a.Y + (int64_t)s0 * NPTS * NV * NV);
        for (int i = tid; i < ns * NPTS * NV * WR; i += CT)
            *reinterpret_cast<unsigned *>(sl + (size_t)(i / WR) * P::LROW + (i % WR) * 4) = src[i];
    }
    // dst = A pub on the CTA's sites (pub published and a grid barrier passed)
    auto apply = [&](C<R> *dst) {
        for (int i = tid; i < ns * NPTS * NV; i += CT) {
            const int l = i % NV, sd = i / NV, d = sd % NPTS, site = s0 + sd / NPTS;
            const int o = d > 0 ? a.nbr[(int64_t)site * (NPTS - 1) + d - 1] : site;
            sin[i] = __ldcg(pub + (int64_t)o * NV + l);
        }
        __syncthreads();
        for (int i = tid; i < ns * NPTS * NV; i += CT) {
            const unsigned char *row = cached ? sl + (size_t)i * P::LROW
                                              : reinterpret_cast<const unsigned char *>(a.Y + ((int64_t)s0 * NPTS * NV + i) * NV);
            sp[i] = row_times<R, LT, NV>(row, sin + i / NV * NV);
        }
        __syncthreads();
        for (int e = tid; e < own; e += CT) {
            const int site = e / NV, k = e - site * NV;
            C<R> t[4];
#pragma unroll
            for (int d = 0; d < NPTS - 1; ++d) {
                const C<R> v = sp[(site * NPTS + d + 1) * NV + k];
                t[d % 4] = d < 4 ? v : t[d % 4] + v;
            }
            dst[e] = sp[site * NPTS * NV + k] + pair_sum<4>(t);
        }
        __syncthreads();
    };
    // tot[i] = the sum over all CTAs of <u_i, v_i>, i < n, u_i and v_i given by
    // the index; the partials in region `reg`, which no CTA reads any more
    // (sums of the type of `zero`)
    auto reduce = [&](auto zero, int n, int reg, auto u, auto v) {
        using S = decltype(zero);
        AccC<S> *pr = reinterpret_cast<AccC<S> *>(a.part) + (size_t)reg * (MAXR + 2) * nb;
        for (int i = warp; i < n; i += CT / 32) {
            const C<R> *ui = u(i), *vi = v(i);
            AccC<S> s;
            acc_init(s.re);
            acc_init(s.im);
            for (int e = lane; e < own; e += 32) {
                const C<R> p = ui[e], q = vi[e];
                acc_fma(s.re, p.x, q.x);
                acc_fma(s.re, p.y, q.y);
                acc_fma(s.im, p.x, q.y);
                acc_fma(s.im, -p.y, q.x);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                acc_add(s.re, acc_xor(s.re, o));
                acc_add(s.im, acc_xor(s.im, o));
            }
            if (lane == 0) pr[(size_t)i * nb + blockIdx.x] = s;
        }
        __threadfence();
        grid.sync();
        for (int i = warp; i < n; i += CT / 32) {
            AccC<S> s;
            acc_init(s.re);
            acc_init(s.im);
            for (int k = lane; k < nb; k += 32) {
                const float4 w = __ldcg(reinterpret_cast<const float4 *>(pr + (size_t)i * nb + k));
                const AccC<S> t = *reinterpret_cast<const AccC<S> *>(&w);
                acc_add(s.re, t.re);
                acc_add(s.im, t.im);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                acc_add(s.re, acc_xor(s.re, o));
                acc_add(s.im, acc_xor(s.im, o));
            }
            if (lane == 0) tot[i] = make_double2(acc_value(s.re), acc_value(s.im));
        }
        __syncthreads();
    };

    for (int e = tid; e < own; e += CT) {
        x[e] = mk<R>(0, 0);
        const C<R> v = a.b[e0 + e];
        r[e] = v;
        pub[e0 + e] = v;
    }
    __syncthreads();
    reduce(0.0, 1, 0, [&](int) { return r; }, [&](int) { return r; });
    double bn2 = tot[0].x;
    // FP32 fields: the solve runs on b scaled by the power of two that brings |b|
    // near 1, so that the FP32 products above neither vanish nor overflow
    // whatever b's size; x is scaled back at the end (both exact)
    R up = 1, down = 1, up2 = 1, down2 = 1;  // each in two factors, which FP32 holds
    if (sizeof(R) == 4 && bn2 > 0.0 && isfinite(bn2)) {
        const int e = ((__double2hiint(bn2) >> 20) - 1023) >> 1, h = e >> 1;  // |b|^2 is no FP64 denormal
        auto pow2 = [](int n) { return (R)__int_as_float((n + 127) << 23); };
        up = pow2(-h);
        up2 = pow2(h - e);
        down = pow2(h);
        down2 = pow2(e - h);
        bn2 *= __hiloint2double((1023 - 2 * e) << 20, 0);
        for (int i = tid; i < own; i += CT) pub[e0 + i] = r[i] = up2 * (up * r[i]);
    }
    double rn2 = bn2;
    int it = 0, k = 0;
    if (bn2 > 0.0) {
        const double stop = a.tol * a.tol * bn2;
        while (it < a.maxiter && rn2 > stop) {
            C<R> *w = W(k), *z = Z(k);
            for (int e = tid; e < own; e += CT) z[e] = r[e];
            __threadfence();
            grid.sync();  // pub = r everywhere
            apply(w);
            // values 0 .. k-1: <W_i, w>; k: |w|^2; k + 1: <w, r>
            auto U = [&](int i) { return i < k ? W(i) : w; };
            auto V = [&](int i) { return i <= k ? w : r; };
            double ww = 0.0, wrx = 0.0, wry = 0.0;
            for (int pass = 0; pass < 2; ++pass) {
                reduce(A{}, k + 2, pass, U, V);
                ww = tot[k].x;
                wrx = tot[k + 1].x;
                wry = tot[k + 1].y;
                if (k == 0) break;
                double removed = 0.0;
                for (int i = 0; i < k; ++i) removed += tot[i].x * tot[i].x + tot[i].y * tot[i].y;
                for (int e = tid; e < own; e += CT) {
                    C<R> wv = w[e], zv = z[e];
                    for (int i = 0; i < k; ++i) {
                        const C<R> m = mk<R>(-(R)tot[i].x, -(R)tot[i].y);
                        cadd_prod(wv, m, W(i)[e]);
                        cadd_prod(zv, m, Z(i)[e]);
                    }
                    w[e] = wv;
                    z[e] = zv;
                }
                __syncthreads();  // tot is rewritten by the next reduction
                const bool again = pass == 0 && removed >= 0.1 * ww;
                ww -= removed;
                if (!again) break;
            }
            if (!(ww > 0.0)) break;  // breakdown: same decision in every CTA
            const double inv = 1.0 / sqrt(ww), ar = wrx * inv, ai = wry * inv;
            const R sc = (R)inv;
            const C<R> al = mk<R>((R)ar, (R)ai), mal = mk<R>(-(R)ar, -(R)ai);
            for (int e = tid; e < own; e += CT) {
                const C<R> zv = sc * z[e], wv = sc * w[e];
                C<R> xv = x[e], rv = r[e];
                cadd_prod(xv, al, zv);
                cadd_prod(rv, mal, wv);
                z[e] = zv;
                w[e] = wv;
                x[e] = xv;
                r[e] = rv;
                pub[e0 + e] = rv;  // every CTA is past its reading of pub (the reduction's barrier)
            }
            rn2 -= ar * ar + ai * ai;
            ++it;
            ++k;
            __syncthreads();
            if (k == a.restart || rn2 <= stop) {
                // true residual r = b - A x
                for (int e = tid; e < own; e += CT) pub[e0 + e] = x[e];
                __threadfence();
                grid.sync();
                apply(r);
                for (int e = tid; e < own; e += CT) {
                    const C<R> v = a.b[e0 + e];
                    r[e] = up2 * (up * v) - r[e];
                }
                __syncthreads();
                reduce(A{}, 1, 0, [&](int) { return r; }, [&](int) { return r; });
                for (int e = tid; e < own; e += CT) pub[e0 + e] = r[e];
                rn2 = tot[0].x;
                k = 0;
                __syncthreads();
            }
        }
    }
    for (int e = tid; e < own; e += CT) a.x[e0 + e] = down2 * (down * x[e]);
    if (blockIdx.x == 0 && tid == 0) atomicAdd(a.iters, it);
}

// Whole sites per CTA, one CTA per SM: the vectors' slices in shared memory
// where 2 restart + 2 of them and two stages of the stencil's inputs fit, the
// links with them where those fit too.
template <typename R, typename LT, int NV, int NPTS> void launch_nv(dwf_ctx *c, Args<R, LT> &a, int max_ctas) {
    const SmemPlan<R, LT, NV, NPTS> plan(a.g.V, a.restart, max_ctas, (size_t)c->smem_optin - 4096);
    if (plan.total <= (size_t)c->smem_optin - 4096) {
        void *fn = (void *)coarse_gcr_smem_kernel<R, LT, NV, NPTS>;
        // one value whatever this launch needs: the lattices of a batch launch
        // from several threads, and the limit belongs to the kernel
        DWF_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, c->smem_optin - 4096));
        int spc = (int)plan.spc, cached = plan.cached ? 1 : 0;
        void *kargs[] = {&a, &spc, &cached};
        DWF_CUDA(coop_launch(c, fn, dim3((unsigned)((a.g.V + spc - 1) / spc)), dim3(CT), kargs, plan.total));
        return;
    }
    void *kargs[] = {&a};
    const int64_t nblk = std::max<int64_t>(1, std::min<int64_t>((a.g.V * NV + CT - 1) / CT, max_ctas));
    void *fn = (void *)coarse_gcr_kernel<R, LT, NV, NPTS>;
    int per_sm = 0;
    DWF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, CT, 0));
    DWF_REQUIRE(per_sm >= 1, DWF_ECUDA, "fused coarse solver cannot be co-resident");
    DWF_CUDA(coop_launch(c, fn, dim3((unsigned)nblk), dim3(CT), kargs, 0));
}

// Launch the solver for a stencil of NPTS points (9: R D P; 33: the squared
// operator's P^+ D^+ D P) on at most max_ctas CTAs.
template <typename R, typename LT, int NPTS>
void launch_t(dwf_ctx *c, const Level &L, const LT *Y, C<R> *x, const C<R> *b, C<R> *r, C<R> *Z, C<R> *W,
                     double2 *part, int *iters, double tol, int maxiter, int restart, int max_ctas) {
    Args<R, LT> a;
    a.Y = Y;
    a.nbr = L.nbr.as<int>();
    a.g = L.lg.g;
    a.b = b;
    a.x = x;
    a.r = r;
    a.Z = Z;
    a.W = W;
    a.part = part;
    a.tol = tol;
    a.maxiter = maxiter;
    a.restart = restart;
    a.iters = iters;
    switch (L.lg.ncomp) {
        case 2: launch_nv<R, LT, 2, NPTS>(c, a, max_ctas); break;
        case 4: launch_nv<R, LT, 4, NPTS>(c, a, max_ctas); break;
        case 6: launch_nv<R, LT, 6, NPTS>(c, a, max_ctas); break;
        case 8: launch_nv<R, LT, 8, NPTS>(c, a, max_ctas); break;
        case 12: launch_nv<R, LT, 12, NPTS>(c, a, max_ctas); break;
        case 16: launch_nv<R, LT, 16, NPTS>(c, a, max_ctas); break;
        case 24: launch_nv<R, LT, 24, NPTS>(c, a, max_ctas); break;
        case 32: launch_nv<R, LT, 32, NPTS>(c, a, max_ctas); break;
        default: throw Error{DWF_EINVAL, "unsupported Nvec"};
    }
    DWF_CHECK_LAUNCH();
}

}  // namespace

}  // namespace dwf
