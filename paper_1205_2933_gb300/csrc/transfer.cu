// Block transfer operators (Sec. 1: restrictor R and prolongator P with
// R P = 1_c; Sec. 2: near-null vectors cut into blocks, the blocks cover the
// whole fifth dimension).
//
// A coarse site owns a block of bx*by*bz*bt sites of the finer level with all
// their components and all s.  In the s-fastest layout the elements of one
// finer site are contiguous (ncomp*Ls of them), so a CTA that walks the
// block site by site reads whole contiguous runs.  One CTA per coarse site;
// reductions over the block use warp shuffles, then shared memory.
#include <cooperative_groups.h>

#include "mg.cuh"

namespace dwf {

namespace cg = cooperative_groups;

namespace {

// n / d for 0 <= n < 2^31 as a multiply-high, an addition and a shift
struct FastDiv {
    unsigned m;
    int l, d;
    __device__ __forceinline__ unsigned div(unsigned n) const { return (__umulhi(m, n) + n) >> l; }
};

FastDiv fast_div(int d) {
    FastDiv f{0, 0, d};
    while (((int64_t)1 << f.l) < d) ++f.l;
    f.m = (unsigned)((((uint64_t)1 << 32) * (((uint64_t)1 << f.l) - (uint64_t)d)) / (uint64_t)d + 1);
    return f;
}

struct BlockMap {
    int L[4];        // finer lattice
    int b[4];        // block
    int Lc[4];       // coarse lattice
    int run;         // contiguous elements per finer site = ncomp * Ls
    int64_t bsites;  // sites per block
    int64_t nelem;   // elements per finer field
    FastDiv drun, db[3];
};

// site index of the first finer site of block xc
__device__ __forceinline__ int64_t block_origin(const BlockMap &m, int64_t xc) {
    int64_t t = xc;
    const int c0 = (int)(t % m.Lc[0]); t /= m.Lc[0];
    const int c1 = (int)(t % m.Lc[1]); t /= m.Lc[1];
    const int c2 = (int)(t % m.Lc[2]), c3 = (int)(t / m.Lc[2]);
    return (((int64_t)c3 * m.b[3] * m.L[2] + c2 * m.b[2]) * m.L[1] + c1 * m.b[1]) * m.L[0] + c0 * m.b[0];
}

// address of element e of the block whose first site is `origin`
__device__ __forceinline__ int64_t block_elem(const BlockMap &m, int64_t origin, unsigned e) {
    unsigned i = m.drun.div(e);
    const unsigned rem = e - i * m.run;
    unsigned q = m.db[0].div(i);
    const unsigned o0 = i - q * m.b[0];
    i = q;
    q = m.db[1].div(i);
    const unsigned o1 = i - q * m.b[1];
    i = q;
    q = m.db[2].div(i);
    const unsigned o2 = i - q * m.b[2];
    return (origin + (((int64_t)q * m.L[2] + o2) * m.L[1] + o1) * m.L[0] + o0) * m.run + rem;
}

__device__ __forceinline__ int64_t block_elem_addr(const BlockMap &m, int64_t xc, int64_t e) {
    int64_t i = e / m.run;
    int rem = (int)(e - i * m.run);
    int c[4], o[4];
    int64_t t = xc;
    c[0] = (int)(t % m.Lc[0]); t /= m.Lc[0];
    c[1] = (int)(t % m.Lc[1]); t /= m.Lc[1];
    c[2] = (int)(t % m.Lc[2]); c[3] = (int)(t / m.Lc[2]);
    o[0] = (int)(i % m.b[0]); i /= m.b[0];
    o[1] = (int)(i % m.b[1]); i /= m.b[1];
    o[2] = (int)(i % m.b[2]); o[3] = (int)(i / m.b[2]);
    int64_t site = (((int64_t)(c[3] * m.b[3] + o[3]) * m.L[2] + (c[2] * m.b[2] + o[2])) * m.L[1] +
                    (c[1] * m.b[1] + o[1])) * m.L[0] + (c[0] * m.b[0] + o[0]);
    return site * m.run + rem;
}

BlockMap make_map(const Level &L) {
    BlockMap m;
    for (int i = 0; i < 4; ++i) {
        m.L[i] = L.lg.g.L[i];
        m.b[i] = L.block[i];
        m.Lc[i] = m.L[i] / m.b[i];
    }
    m.run = L.lg.ncomp * L.lg.g.Ls;
    m.bsites = (int64_t)m.b[0] * m.b[1] * m.b[2] * m.b[3];
    m.nelem = L.lg.nelem;
    m.drun = fast_div(m.run);
    for (int i = 0; i < 3; ++i) m.db[i] = fast_div(m.b[i]);
    return m;
}

int64_t ncoarse(const BlockMap &m) { return (int64_t)m.Lc[0] * m.Lc[1] * m.Lc[2] * m.Lc[3]; }

constexpr int TT = 256;  // threads per CTA of the block kernels

// ---- restriction and prolongation -----------------------------------------
//
// Both read the basis once per call and up to 12 right-hand sides; a block is
// cut into pieces so that small coarse lattices fill the chip as well (one
// CTA per coarse site left 16 to 108 of them on 152 SMs).

// EPP consecutive elements travel as one access (a site's run is even): 16
// bytes of an FP32 or FP64 field, 8 bytes of the FP16 basis.
template <typename R, typename QT> struct Piece;
template <> struct Piece<float, float2> {
    static constexpr int EPP = 2;
    using FP = float4;
    using QP = float4;
    static __device__ __forceinline__ void q(const QP &v, float2 o[2]) { o[0] = make_float2(v.x, v.y); o[1] = make_float2(v.z, v.w); }
};
template <> struct Piece<float, __half2> {
    static constexpr int EPP = 2;
    using FP = float4;
    using QP = uint2;
    static __device__ __forceinline__ void q(const QP &v, float2 o[2]) {
        o[0] = __half22float2(*reinterpret_cast<const __half2 *>(&v.x));
        o[1] = __half22float2(*reinterpret_cast<const __half2 *>(&v.y));
    }
};
template <> struct Piece<double, double2> {
    static constexpr int EPP = 1;
    using FP = double2;
    using QP = double2;
    static __device__ __forceinline__ void q(const QP &v, double2 o[1]) { o[0] = v; }
};
__device__ __forceinline__ void unpiece(const float4 &v, float2 o[2]) { o[0] = make_float2(v.x, v.y); o[1] = make_float2(v.z, v.w); }
__device__ __forceinline__ void unpiece(const double2 &v, double2 o[1]) { o[0] = v; }
__device__ __forceinline__ float4 piece(const float2 o[2]) { return make_float4(o[0].x, o[0].y, o[1].x, o[1].y); }
__device__ __forceinline__ double2 piece(const double2 o[1]) { return o[0]; }

// How a restriction CTA (8 warps) shares its work: RG groups of KG basis rows
// times RC groups of NB right-hand sides times EH parts of the elements.  A
// lane keeps KG x NB sums; KG NB is at most 36 (FP32) or 16 (FP64) for the
// registers.  SE elements of all rows make one stage in shared memory.
constexpr bool restrict_fits(int rg, int nv, int nb, int rc, int lim) {
    return nv % rg == 0 && (nv / rg) * nb <= lim && nv / rg <= 12 && rg * rc <= 8;
}
constexpr int restrict_groups(int nv, int nb, int rc, int lim) {  // RG, or 0 where nothing fits
    for (int rg = 1; rg <= 8; rg *= 2)
        if (restrict_fits(rg, nv, nb, rc, lim)) return rg;
    return 0;
}
template <typename R, typename QT, int NV, int NB, int RC> struct RShape {
    static constexpr int RG = restrict_groups(NV, NB, RC, sizeof(R) == 8 ? 16 : 36);
    static constexpr int KG = NV / RG;
    static constexpr int EH = 8 / (RG * RC);
    static constexpr int RT = NB * RC;
    static constexpr int EPP = Piece<R, QT>::EPP;
    static constexpr int SE = 32 * EPP * EH;
    static constexpr size_t stage = (sizeof(QT) * NV + sizeof(C<R>) * RT) * SE;
    static constexpr int NS = 100 * 1024 / stage >= 4 ? 4 : 100 * 1024 / stage >= 3 ? 3 : 2;
    static constexpr size_t red = sizeof(C<R>) * (EH + 1) * RT * NV;
    static constexpr size_t smem = stage * NS > red ? stage * NS : red;
};

template <int BYTES> __device__ __forceinline__ void cp_async(void *dst, const void *src, bool on) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = on ? BYTES : 0;  // 0: the destination is filled with zeros
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(d), "l"(src), "n"(BYTES), "r"(n) : "memory");
}

// c_r(xc, k) = sum_e conj(Q_k(e)) f_r(e), k < NV, for the NB*RC right-hand
// sides of one group (zeros beyond nrhs).  A cluster of CS CTAs shares one
// coarse site; each runs over a part of the block's elements in NS stages of
// asynchronous copies and the cluster's first CTA adds the parts in a fixed
// order through distributed shared memory.  Bound: reading the basis once
// (FP32, 12 right-hand sides: the FMA pipe comes close, 8 NV nrhs flops per
// element); the loop is 12 shared loads of 16 bytes for 288 FMAs per lane at
// Nvec 24.  12 right-hand sides, Nvec 24, Ls 16, 4^4 blocks:
// 0.42 ms for 12^3 x 16 (1.5 GB read: 3.6 TB/s) against 1.37 ms with one CTA
// per site and four right-hand sides and loads in the loop; one right-hand
// side at 8^3 x 16 (32 sites) 54 us against 429 us
template <typename R, typename QT, int NV, int NB, int RC>
__global__ void __launch_bounds__(TT, 2) restrict_kernel(C<R> *__restrict__ cout, const C<R> *__restrict__ f,
                                                         const QT *__restrict__ Q, BlockMap m, int nrhs, int ngroups,
                                                         int per, int64_t cstride) {
    using S = RShape<R, QT, NV, NB, RC>;
    using P = Piece<R, QT>;
    constexpr int KG = S::KG, EH = S::EH, EPP = S::EPP, SE = S::SE, NS = S::NS, RT = S::RT;
    constexpr int PIECES = 32 * EH, ROWSTEP = TT / PIECES;
    extern __shared__ __align__(16) unsigned char smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned cs = cluster.num_blocks(), rank = cluster.block_rank();
    const int64_t id = blockIdx.x / cs;
    const int64_t xc = id / ngroups;
    const int r0 = (int)(id - xc * ngroups) * per;
    const int nr = min(per, nrhs - r0);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wk = warp % S::RG, wr = (warp / S::RG) % RC, we = warp / (S::RG * RC);
    const unsigned ne = (unsigned)(m.bsites * m.run);
    const unsigned nst = (ne + SE - 1) / SE;                  // stages of the whole block
    const unsigned spc = (nst + cs - 1) / cs;                 // ... of one CTA
    const unsigned st0 = rank * spc, st1 = min(nst, st0 + spc);
    const int64_t origin = block_origin(m, xc);

    auto stage_q = [&](int s) { return reinterpret_cast<QT *>(smem + S::stage * s); };
    auto stage_f = [&](int s) { return reinterpret_cast<C<R> *>(smem + S::stage * s + sizeof(QT) * NV * SE); };
    auto fill = [&](unsigned st) {
        if (st < st1) {
            const int pc = threadIdx.x % PIECES;
            const unsigned e = st * SE + pc * EPP;
            const bool in = e < ne;
            const int64_t ad = in ? block_elem(m, origin, e) : 0;
            QT *sq = stage_q(st % NS) + pc * EPP;
            C<R> *sf = stage_f(st % NS) + pc * EPP;
            for (int row = threadIdx.x / PIECES; row < NV; row += ROWSTEP)
                cp_async<(int)sizeof(typename P::QP)>(sq + row * SE, Q + (int64_t)row * m.nelem + ad, in);
            for (int row = threadIdx.x / PIECES; row < RT; row += ROWSTEP) {
                const bool on = in && row < nr;
                cp_async<16>(sf + row * SE, f + (int64_t)(r0 + (on ? row : 0)) * m.nelem + ad, on);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };

    C<R> acc[KG][NB];
#pragma unroll
    for (int a = 0; a < KG; ++a)
#pragma unroll
        for (int r = 0; r < NB; ++r) acc[a][r] = mk<R>(0, 0);
#pragma unroll
    for (int i = 0; i < NS - 1; ++i) fill(st0 + i);
    for (unsigned st = st0; st < st1; ++st) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(NS - 2) : "memory");
        __syncthreads();
        fill(st + NS - 1);
        const int off = (we * 32 + lane) * EPP;
        const QT *sq = stage_q(st % NS) + wk * KG * SE + off;
        const C<R> *sf = stage_f(st % NS) + wr * NB * SE + off;
        C<R> q[KG][EPP];
#pragma unroll
        for (int a = 0; a < KG; ++a) P::q(*reinterpret_cast<const typename P::QP *>(sq + a * SE), q[a]);
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            C<R> v[EPP];
            unpiece(*reinterpret_cast<const typename P::FP *>(sf + r * SE), v);
#pragma unroll
            for (int a = 0; a < KG; ++a)
#pragma unroll
                for (int x = 0; x < EPP; ++x) cfmac(acc[a][r], q[a][x], v[x]);
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    // part sums [EH][RT][NV], then this CTA's [RT][NV] behind them
    C<R> *red = reinterpret_cast<C<R> *>(smem);
    C<R> *mine = red + EH * RT * NV;
#pragma unroll
    for (int a = 0; a < KG; ++a)
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            C<R> v = acc[a][r];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
                v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
            }
            if (lane == 0) red[(we * RT + wr * NB + r) * NV + wk * KG + a] = v;
        }
    __syncthreads();
    for (int i = threadIdx.x; i < RT * NV; i += TT) {
        C<R> v = red[i];
#pragma unroll
        for (int h = 1; h < EH; ++h) v = v + red[h * RT * NV + i];
        mine[i] = v;
    }
    cluster.sync();
    if (rank == 0)
        for (int i = threadIdx.x; i < nr * NV; i += TT) {
            C<R> v = mine[i];
            for (unsigned h = 1; h < cs; ++h) v = v + cluster.map_shared_rank(mine, h)[i];
            cout[(int64_t)(r0 + i / NV) * cstride + xc * NV + i % NV] = v;
        }
    cluster.sync();  // the parts stay readable until the first CTA has added them
}

// f_r(e) (+)= sum_k Q_k(e) c_r(xc, k) for NB right-hand sides from r0 on (those
// below nrhs are written).  grid.x = coarse sites x pieces of a block; a
// thread owns EPP elements, keeps NB sums for each and streams over the basis
// rows, whose loads do not depend on one another; the coefficients are
// broadcast from shared memory, two right-hand sides per load.  Bound by
// reading the basis and writing the fields: 0.35 ms for 12 right-hand sides,
// Nvec 24, at 12^3 x 16 x 16 (0.70 ms with one CTA per site), 49 us for one at
// 8^3 x 16 x 16 (608 us)
template <typename R, typename QT, int NV, int NB>
__global__ void __launch_bounds__(TT, 2) prolong_kernel(C<R> *__restrict__ f, const C<R> *__restrict__ cin,
                                                     const QT *__restrict__ Q, BlockMap m, int nrhs, int r0,
                                                     int64_t cstride, int pieces, int accumulate) {
    using P = Piece<R, QT>;
    constexpr int EPP = P::EPP;
    __shared__ __align__(16) C<R> cs[NV][NB];
    const int64_t xc = blockIdx.x / pieces;
    const unsigned part = blockIdx.x - (unsigned)xc * pieces;
    const int nr = min(NB, nrhs - r0);
    for (int i = threadIdx.x; i < NV * NB; i += TT) {
        const int k = i / NB, r = i - k * NB;
        cs[k][r] = r < nr ? cin[(int64_t)(r0 + r) * cstride + xc * NV + k] : mk<R>(0, 0);
    }
    __syncthreads();
    const unsigned ne = (unsigned)(m.bsites * m.run);
    const int64_t origin = block_origin(m, xc);
    f += (int64_t)r0 * m.nelem;
    for (unsigned e = (part * TT + threadIdx.x) * EPP; e < ne; e += (unsigned)pieces * TT * EPP) {
        const int64_t a = block_elem(m, origin, e);
        C<R> v[NB][EPP];
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            if (accumulate && r < nr)
                unpiece(*reinterpret_cast<const typename P::FP *>(f + (int64_t)r * m.nelem + a), v[r]);
            else
#pragma unroll
                for (int x = 0; x < EPP; ++x) v[r][x] = mk<R>(0, 0);
        }
        constexpr int KU = NB >= 6 ? (NV % 4 == 0 ? 4 : 2) : NV % 8 == 0 ? 8 : NV % 6 == 0 ? 6 : NV;
#pragma unroll 1
        for (int k0 = 0; k0 < NV; k0 += KU) {
            typename P::QP w[KU];
#pragma unroll
            for (int k = 0; k < KU; ++k)
                w[k] = *reinterpret_cast<const typename P::QP *>(Q + (int64_t)(k0 + k) * m.nelem + a);
#pragma unroll
            for (int k = 0; k < KU; ++k) {
                C<R> q[EPP];
                P::q(w[k], q);
#pragma unroll
                for (int r = 0; r < NB; ++r)
#pragma unroll
                    for (int x = 0; x < EPP; ++x) cfma(v[r][x], q[x], cs[k0 + k][r]);
            }
        }
#pragma unroll
        for (int r = 0; r < NB; ++r)
            if (r < nr) *reinterpret_cast<typename P::FP *>(f + (int64_t)r * m.nelem + a) = piece(v[r]);
    }
}

// G[xc][k][l] = sum_{e in block} conj(A_k(e)) B_l(e), FP64 accumulation.
// Chunks of CH elements of all NV fields of A and B are staged in shared
// memory; each thread owns a few (k,l) pairs.
template <typename R, int NV, int CH>
__global__ void __launch_bounds__(TT) gram_kernel(double2 *__restrict__ G, const C<R> *__restrict__ A,
                                                  const C<R> *__restrict__ B, BlockMap m) {
    __shared__ C<R> sA[NV][CH];
    __shared__ C<R> sB[NV][CH];
    constexpr int NP = NV * NV;
    constexpr int PPT = (NP + TT - 1) / TT;
    const int64_t xc = blockIdx.x;
    const int64_t ne = m.bsites * m.run;
    double2 acc[PPT];
#pragma unroll
    for (int q = 0; q < PPT; ++q) acc[q] = make_double2(0, 0);
    for (int64_t e0 = 0; e0 < ne; e0 += CH) {
        for (int j = threadIdx.x; j < NV * CH; j += TT) {
            int k = j / CH, e = j - k * CH;
            C<R> a = mk<R>(0, 0), b = mk<R>(0, 0);
            if (e0 + e < ne) {
                int64_t ad = block_elem_addr(m, xc, e0 + e);
                a = A[k * m.nelem + ad];
                b = B[k * m.nelem + ad];
            }
            sA[k][e] = a;
            sB[k][e] = b;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < PPT; ++q) {
            int p = threadIdx.x + q * TT;
            if (p < NP) {
                int k = p / NV, l = p - k * NV;
                C<R> s = mk<R>(0, 0);
#pragma unroll 8
                for (int e = 0; e < CH; ++e) cfmac(s, sA[k][e], sB[l][e]);
                acc[q].x += (double)s.x;
                acc[q].y += (double)s.y;
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < PPT; ++q) {
        int p = threadIdx.x + q * TT;
        if (p < NP) G[xc * NP + p] = acc[q];
    }
}

// Cholesky G = R^+ R (R upper triangular, positive diagonal) and Rinv = R^-1,
// one thread per coarse site, in FP64.  info[xc] = 0 or (1 + failing column).
__global__ void chol_inv_kernel(const double2 *__restrict__ G, double2 *__restrict__ Rm,
                                double2 *__restrict__ Ri, int *info, int64_t nc, int nv) {
    int64_t xc = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (xc >= nc) return;
    const double2 *g = G + xc * nv * nv;
    double2 *r = Rm + xc * nv * nv;
    double2 *ri = Ri + xc * nv * nv;
    int bad = 0;
    for (int i = 0; i < nv * nv; ++i) { r[i] = make_double2(0, 0); ri[i] = make_double2(0, 0); }
    for (int j = 0; j < nv && !bad; ++j) {
        double d = g[j * nv + j].x;
        for (int i = 0; i < j; ++i) d -= r[i * nv + j].x * r[i * nv + j].x + r[i * nv + j].y * r[i * nv + j].y;
        if (!(d > 1e-28 * fabs(g[j * nv + j].x)) || !(d > 0.0)) { bad = j + 1; break; }
        double rd = sqrt(d);
        r[j * nv + j] = make_double2(rd, 0);
        for (int k = j + 1; k < nv; ++k) {
            double2 s = g[j * nv + k];
            for (int i = 0; i < j; ++i) {
                double2 t = cmulc(r[i * nv + j], r[i * nv + k]);
                s.x -= t.x;
                s.y -= t.y;
            }
            r[j * nv + k] = make_double2(s.x / rd, s.y / rd);
        }
    }
    info[xc] = bad;
    if (bad) return;
    // back substitution: R X = I, X upper triangular
    for (int col = 0; col < nv; ++col) {
        for (int i = col; i >= 0; --i) {
            double2 s = make_double2(i == col ? 1.0 : 0.0, 0.0);
            for (int k = i + 1; k <= col; ++k) {
                double2 t = cmul(r[i * nv + k], ri[k * nv + col]);
                s.x -= t.x;
                s.y -= t.y;
            }
            double dinv = 1.0 / r[i * nv + i].x;
            ri[i * nv + col] = make_double2(s.x * dinv, s.y * dinv);
        }
    }
}

// Q_l <- sum_{k <= l} Q_k Rinv[k][l] in place, per block.
template <typename R, int NV>
__global__ void __launch_bounds__(TT) apply_rinv_kernel(C<R> *__restrict__ Q, const double2 *__restrict__ Ri, BlockMap m) {
    __shared__ C<R> r[NV * NV];
    const int64_t xc = blockIdx.x;
    for (int i = threadIdx.x; i < NV * NV; i += TT) r[i] = cvt<C<R>, double2>(Ri[xc * NV * NV + i]);
    __syncthreads();
    const int64_t ne = m.bsites * m.run;
    for (int64_t e = threadIdx.x; e < ne; e += TT) {
        int64_t a = block_elem_addr(m, xc, e);
        C<R> v[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] = Q[k * m.nelem + a];
#pragma unroll
        for (int l = NV - 1; l >= 0; --l) {
            C<R> s = mk<R>(0, 0);
#pragma unroll
            for (int k = 0; k <= l; ++k) cfma(s, v[k], r[k * NV + l]);
            Q[l * m.nelem + a] = s;
        }
    }
}

// Gamma split of adaptive vectors into Q (see mg.cuh).
template <typename R>
__global__ void gamma_split_kernel(C<R> *__restrict__ Q, const double2 *__restrict__ v, int nadapt, int split,
                                   int64_t nelem, int ncomp, int Ls, int fine) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nelem; i += (int64_t)gridDim.x * blockDim.x) {
        int s = (int)(i % Ls);
        int64_t sc = i / Ls;
        int comp = (int)(sc % ncomp);
        int64_t site = sc / ncomp;
        for (int j = 0; j < nadapt; ++j) {
            double2 a = v[j * nelem + i];
            if (!split) {
                Q[j * nelem + i] = cvt<C<R>, double2>(a);
                continue;
            }
            double2 ga;  // (Gamma v)(i)
            if (fine) {
                double2 b = v[j * nelem + (site * ncomp + comp) * Ls + (Ls - 1 - s)];
                double g5 = comp < 6 ? 1.0 : -1.0;
                ga = make_double2(g5 * b.x, g5 * b.y);
            } else {
                double gc = (comp & 1) ? -1.0 : 1.0;
                ga = make_double2(gc * a.x, gc * a.y);
            }
            Q[(2 * j) * nelem + i] = cvt<C<R>, double2>(make_double2(0.5 * (a.x + ga.x), 0.5 * (a.y + ga.y)));
            Q[(2 * j + 1) * nelem + i] = cvt<C<R>, double2>(make_double2(0.5 * (a.x - ga.x), 0.5 * (a.y - ga.y)));
        }
    }
}

#define NV_DISPATCH(nv, MACRO)                                      \
    switch (nv) {                                                   \
        case 2: MACRO(2); break;                                    \
        case 4: MACRO(4); break;                                    \
        case 6: MACRO(6); break;                                    \
        case 8: MACRO(8); break;                                    \
        case 12: MACRO(12); break;                                  \
        case 16: MACRO(16); break;                                  \
        case 24: MACRO(24); break;                                  \
        case 32: MACRO(32); break;                                  \
        default: throw Error{DWF_EINVAL, "unsupported Nvec (use 2,4,6,8,12,16,24,32)"}; \
    }

}  // namespace

namespace {

template <typename R, typename QT, int NV, int NB, int RC>
void restrict_launch(dwf_ctx *c, C<R> *cout, const C<R> *f, const QT *Q, const BlockMap &m, int nrhs, int ngroups,
                     int per) {
    using S = RShape<R, QT, NV, NB, RC>;
    auto *fn = restrict_kernel<R, QT, NV, NB, RC>;
    const int64_t nc = ncoarse(m), clusters = nc * ngroups;
    const int64_t stages = (m.bsites * m.run + S::SE - 1) / S::SE;
    int cs = 1;
    while (cs < 8 && clusters * cs < 2 * (int64_t)c->sm_count && stages >= 4 * cs) cs *= 2;
    DWF_REQUIRE(clusters * cs < ((int64_t)1 << 31) && m.bsites * m.run < ((int64_t)1 << 30), DWF_EINVAL,
                "restriction grid too large");
    if (S::smem > 48 * 1024)
        DWF_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem));
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)cs;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(clusters * cs));
    cfg.blockDim = dim3(TT);
    cfg.dynamicSmemBytes = S::smem;
    cfg.stream = c->stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    DWF_CUDA(cudaLaunchKernelEx(&cfg, fn, cout, f, Q, m, nrhs, ngroups, per, nc * NV));
    DWF_CHECK_LAUNCH();
}

// Right-hand sides per group: at most 12 (8 at Nvec 32, whose 12 would not fit
// the registers), the groups of equal width; one at a time in FP64 and with
// the FP16 basis, which only the one-right-hand-side V-cycle uses.  Clusters
// grow until the grid has two CTAs per SM (108 sites: 4 CTAs each), as long
// as every CTA keeps at least two stages.
template <typename R, typename QT, int NV>
void restrict_nv(dwf_ctx *c, C<R> *cout, const C<R> *f, const QT *Q, const BlockMap &m, int nrhs) {
    if constexpr (std::is_same<QT, float2>::value) {
        constexpr int most = restrict_groups(NV, 6, 2, 36) ? 12 : 8;
        int ng = (nrhs + most - 1) / most, per = (nrhs + ng - 1) / ng;
        // where clusters of 8 leave SMs with one CTA, two groups per site (the
        // second reads the basis from L2)
        if (per > 6 && ncoarse(m) * ng * 8 < 2 * (int64_t)c->sm_count) {
            ng *= 2;
            per = (nrhs + ng - 1) / ng;
        }
        switch (per) {
            case 1: return restrict_launch<R, QT, NV, 1, 1>(c, cout, f, Q, m, nrhs, ng, per);
            case 2: return restrict_launch<R, QT, NV, 2, 1>(c, cout, f, Q, m, nrhs, ng, per);
            case 3: case 4: return restrict_launch<R, QT, NV, 4, 1>(c, cout, f, Q, m, nrhs, ng, per);
            case 5: case 6: return restrict_launch<R, QT, NV, 6, 1>(c, cout, f, Q, m, nrhs, ng, per);
            case 7: case 8: return restrict_launch<R, QT, NV, 4, 2>(c, cout, f, Q, m, nrhs, ng, per);
            default:
                if constexpr (most == 12) return restrict_launch<R, QT, NV, 6, 2>(c, cout, f, Q, m, nrhs, ng, per);
        }
    } else {
        restrict_launch<R, QT, NV, 1, 1>(c, cout, f, Q, m, nrhs, nrhs, 1);
    }
}

template <typename R, typename QT, int NV, int NB>
void prolong_launch(dwf_ctx *c, C<R> *f, const C<R> *cin, const QT *Q, const BlockMap &m, int nrhs, int r0, bool acc) {
    const int64_t nc = ncoarse(m), ne = m.bsites * m.run;
    const int64_t one = (ne + (int64_t)TT * Piece<R, QT>::EPP - 1) / (TT * Piece<R, QT>::EPP);
    // pieces of a block: one pass over the elements per CTA, several where the
    // grid would exceed 16 CTAs per SM (then the coefficients are staged less often)
    const int64_t want = std::max<int64_t>(1, (16 * (int64_t)c->sm_count + nc - 1) / nc);
    const int pieces = (int)std::min(one, want);
    DWF_REQUIRE(nc * pieces < ((int64_t)1 << 31) && ne < ((int64_t)1 << 30), DWF_EINVAL, "prolongation grid too large");
    prolong_kernel<R, QT, NV, NB><<<(unsigned)(nc * pieces), TT, 0, c->stream>>>(f, cin, Q, m, nrhs, r0, nc * NV, pieces,
                                                                              acc ? 1 : 0);
    DWF_CHECK_LAUNCH();
}

template <typename R, typename QT, int NV>
void prolong_nv(dwf_ctx *c, C<R> *f, const C<R> *cin, const QT *Q, const BlockMap &m, int nrhs, bool acc) {
    if constexpr (std::is_same<QT, float2>::value) {
        const int ng = (nrhs + 11) / 12, per = (nrhs + ng - 1) / ng;
        for (int r0 = 0; r0 < nrhs; r0 += per) {
            const int n = std::min(per, nrhs - r0), end = r0 + n;
            if (n == 1) prolong_launch<R, QT, NV, 1>(c, f, cin, Q, m, end, r0, acc);
            else if (n == 2) prolong_launch<R, QT, NV, 2>(c, f, cin, Q, m, end, r0, acc);
            else if (n <= 4) prolong_launch<R, QT, NV, 4>(c, f, cin, Q, m, end, r0, acc);
            else if (n <= 6) prolong_launch<R, QT, NV, 6>(c, f, cin, Q, m, end, r0, acc);
            else if (n <= 8) prolong_launch<R, QT, NV, 8>(c, f, cin, Q, m, end, r0, acc);
            else prolong_launch<R, QT, NV, 12>(c, f, cin, Q, m, end, r0, acc);
        }
    } else {
        for (int r0 = 0; r0 < nrhs; ++r0) prolong_launch<R, QT, NV, 1>(c, f, cin, Q, m, r0 + 1, r0, acc);
    }
}

template <typename R, typename QT>
void restrict_q(dwf_ctx *c, const Level &L, C<R> *cout, const C<R> *fin, const QT *Q, int nrhs) {
    BlockMap m = make_map(L);
    ProfScope ps(c, K_RESTRICT, nrhs);
#define RK(NV) restrict_nv<R, QT, NV>(c, cout, fin, Q, m, nrhs)
    NV_DISPATCH(L.nv, RK);
#undef RK
}

template <typename R, typename QT>
void prolong_q(dwf_ctx *c, const Level &L, C<R> *fout, const C<R> *cin, const QT *Q, int nrhs, bool acc) {
    BlockMap m = make_map(L);
    ProfScope ps(c, K_PROLONG, nrhs);
#define PK(NV) prolong_nv<R, QT, NV>(c, fout, cin, Q, m, nrhs, acc)
    NV_DISPATCH(L.nv, PK);
#undef PK
}

}  // namespace

template <typename R> void restrict_(dwf_ctx *c, const Level &L, C<R> *cout, const C<R> *fin, const C<R> *Q) {
    restrict_q<R, C<R>>(c, L, cout, fin, Q, 1);
}
template <typename R> void prolong_(dwf_ctx *c, const Level &L, C<R> *fout, const C<R> *cin, const C<R> *Q, bool acc) {
    prolong_q<R, C<R>>(c, L, fout, cin, Q, 1, acc);
}
void restrict_h(dwf_ctx *c, const Level &L, float2 *cout, const float2 *fin, const __half2 *Q) {
    restrict_q<float, __half2>(c, L, cout, fin, Q, 1);
}
void prolong_h(dwf_ctx *c, const Level &L, float2 *fout, const float2 *cin, const __half2 *Q, bool acc) {
    prolong_q<float, __half2>(c, L, fout, cin, Q, 1, acc);
}
template <typename R>
void restrict_batch(dwf_ctx *c, const Level &L, C<R> *cout, const C<R> *fin, const C<R> *Q, int nrhs) {
    restrict_q<R, C<R>>(c, L, cout, fin, Q, nrhs);
}
template <typename R>
void prolong_batch(dwf_ctx *c, const Level &L, C<R> *fout, const C<R> *cin, const C<R> *Q, int nrhs, bool acc) {
    prolong_q<R, C<R>>(c, L, fout, cin, Q, nrhs, acc);
}

namespace {
__global__ void to_half_kernel(__half2 *__restrict__ out, const float2 *__restrict__ in, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = __floats2half2_rn(in[i].x, in[i].y);
}
}  // namespace

template void restrict_batch<float>(dwf_ctx *, const Level &, float2 *, const float2 *, const float2 *, int);
template void restrict_batch<double>(dwf_ctx *, const Level &, double2 *, const double2 *, const double2 *, int);
template void prolong_batch<float>(dwf_ctx *, const Level &, float2 *, const float2 *, const float2 *, int, bool);
template void prolong_batch<double>(dwf_ctx *, const Level &, double2 *, const double2 *, const double2 *, int, bool);

void basis_to_half(dwf_ctx *c, __half2 *out, const float2 *in, int64_t n) {
    unsigned blocks = (unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)c->sm_count * 16);
    to_half_kernel<<<blocks, 256, 0, c->stream>>>(out, in, n);
    DWF_CHECK_LAUNCH();
}

template <typename R> void block_gram(dwf_ctx *c, const Level &L, double2 *G, const C<R> *A, const C<R> *B) {
    BlockMap m = make_map(L);
#define GK(NV) gram_kernel<R, NV, (NV > 16 ? 16 : 32)><<<(unsigned)ncoarse(m), TT, 0, c->stream>>>(G, A, B, m)
    NV_DISPATCH(L.nv, GK);
#undef GK
    DWF_CHECK_LAUNCH();
}

template <typename R> bool block_orthonormalise(dwf_ctx *c, Level &L, C<R> *Q) {
    BlockMap m = make_map(L);
    int64_t nc = ncoarse(m);
    size_t gb = sizeof(double2) * nc * L.nv * L.nv;
    if (L.G.bytes < gb) L.G.alloc(gb);
    if (L.F.bytes < gb) L.F.alloc(gb);
    if (L.Rinv.bytes < gb) L.Rinv.alloc(gb);
    if (L.info.bytes < sizeof(int) * nc) L.info.alloc(sizeof(int) * nc);
    std::vector<int> info(nc);
    for (int pass = 0; pass < 2; ++pass) {  // CholQR2
        block_gram<R>(c, L, L.G.as<double2>(), Q, Q);
        chol_inv_kernel<<<(unsigned)((nc + 63) / 64), 64, 0, c->stream>>>(L.G.as<double2>(), L.F.as<double2>(),
                                                                          L.Rinv.as<double2>(), L.info.as<int>(), nc, L.nv);
        DWF_CHECK_LAUNCH();
        DWF_CUDA(cudaMemcpyAsync(info.data(), L.info.p, sizeof(int) * nc, cudaMemcpyDeviceToHost, c->stream));
        DWF_CUDA(cudaStreamSynchronize(c->stream));
        for (int64_t i = 0; i < nc; ++i)
            if (info[i]) return false;
#define AK(NV) apply_rinv_kernel<R, NV><<<(unsigned)nc, TT, 0, c->stream>>>(Q, L.Rinv.as<double2>(), m)
        NV_DISPATCH(L.nv, AK);
#undef AK
        DWF_CHECK_LAUNCH();
    }
    return true;
}

template <typename R> void gamma_split(dwf_ctx *c, const Level &L, C<R> *Q, const double2 *v, int nadapt, bool split) {
    int64_t n = L.lg.nelem;
    unsigned blocks = (unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)c->sm_count * 16);
    gamma_split_kernel<R><<<blocks, 256, 0, c->stream>>>(Q, v, nadapt, split ? 1 : 0, n, L.lg.ncomp, L.lg.g.Ls,
                                                         L.index == 0 ? 1 : 0);
    DWF_CHECK_LAUNCH();
}

template void restrict_<double>(dwf_ctx *, const Level &, double2 *, const double2 *, const double2 *);
template void restrict_<float>(dwf_ctx *, const Level &, float2 *, const float2 *, const float2 *);
template void prolong_<double>(dwf_ctx *, const Level &, double2 *, const double2 *, const double2 *, bool);
template void prolong_<float>(dwf_ctx *, const Level &, float2 *, const float2 *, const float2 *, bool);
template void block_gram<double>(dwf_ctx *, const Level &, double2 *, const double2 *, const double2 *);
template void block_gram<float>(dwf_ctx *, const Level &, double2 *, const float2 *, const float2 *);
template bool block_orthonormalise<double>(dwf_ctx *, Level &, double2 *);
template bool block_orthonormalise<float>(dwf_ctx *, Level &, float2 *);
template void gamma_split<double>(dwf_ctx *, const Level &, double2 *, const double2 *, int, bool);
template void gamma_split<float>(dwf_ctx *, const Level &, float2 *, const double2 *, int, bool);

}  // namespace dwf
