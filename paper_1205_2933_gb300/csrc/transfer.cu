// Block transfer operators (Sec. 1: restrictor R and prolongator P with
// R P = 1_c; Sec. 2: near-null vectors cut into blocks, the blocks cover the
// whole fifth dimension).
//
// A coarse site owns a block of bx*by*bz*bt sites of the finer level with all
// their components and all s.  In the s-fastest layout the elements of one
// finer site are contiguous (ncomp*Ls of them), so a CTA that walks the
// block site by site reads whole contiguous runs.
#include <cooperative_groups.h>

#include "blockmap.cuh"

namespace dwf {

namespace cg = cooperative_groups;

namespace {

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
// lane keeps KG x NB sums; KG NB is at most 36 (FP32) or 8 (FP64, two chains
// each) for the registers.  SE elements of all rows make one stage in shared memory.
constexpr bool restrict_fits(int rg, int nv, int nb, int rc, int lim) {
    return nv % rg == 0 && (nv / rg) * nb <= lim && nv / rg <= 12 && rg * rc <= 8;
}
constexpr int restrict_groups(int nv, int nb, int rc, int lim) {  // RG, or 0 where nothing fits
    for (int rg = 1; rg <= 8; rg *= 2)
        if (restrict_fits(rg, nv, nb, rc, lim)) return rg;
    return 0;
}
template <typename R, typename QT, int NV, int NB, int RC> struct RShape {
    static constexpr int RG = restrict_groups(NV, NB, RC, sizeof(R) == 8 ? 8 : 36);
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

// c_r(xc, k) = sum_e conj(Q_k(e)) f_r(e), k < NV, for the NB*RC right-hand
// sides of one group (zeros beyond nrhs).  A cluster of CS CTAs shares one
// coarse site; each runs over a part of the block's elements in NS stages of
// asynchronous copies and the cluster's first CTA adds the parts in a fixed
// order through distributed shared memory.  Bound: reading the basis once
// (FP32, 12 right-hand sides: the FMA pipe comes close, 8 NV nrhs flops per
// element); the loop is 12 shared loads of 16 bytes for 288 FMAs and 72 additions
// per lane at Nvec 24.  12 right-hand sides, Nvec 24, Ls 16, 4^4 blocks:
// 0.45 ms for 12^3 x 16 (1.5 GB read: 3.3 TB/s; 0.41 without the additions, see
// the sums below) against 1.37 ms with one CTA
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
            const int64_t ad = in ? box_elem(m.box, origin, e) : 0;
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

    // FP32: the products of a piece are summed first, four roundings at their size
    // and one at that of the running sum instead of four at that.  FP64 (one
    // element per piece, bound by its pipe): the two products of a part in chains
    // of their own, each rounding at a fraction of the sum.
    constexpr int CH = EPP == 1 ? 2 : 1;
    C<R> acc[KG][NB][CH];
#pragma unroll
    for (int a = 0; a < KG; ++a)
#pragma unroll
        for (int r = 0; r < NB; ++r)
#pragma unroll
            for (int h = 0; h < CH; ++h) acc[a][r][h] = mk<R>(0, 0);
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
            for (int a = 0; a < KG; ++a) {
                if constexpr (CH == 2) {
                    cfmac2(acc[a][r][0], acc[a][r][1], q[a][0], v[0]);
                } else {
                    C<R> t = mk<R>(0, 0);
#pragma unroll
                    for (int x = 0; x < EPP; ++x) cfmac(t, q[a][x], v[x]);
                    acc[a][r][0] = acc[a][r][0] + t;
                }
            }
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
            C<R> v = CH == 2 ? acc[a][r][0] + acc[a][r][CH - 1] : acc[a][r][0];
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
// reading the basis and writing the fields: 0.40 ms for 12 right-hand sides,
// Nvec 24, at 12^3 x 16 x 16 (0.70 ms with one CTA per site; 0.35 with one chain of
// multiply-adds per element, which rounds 1.3 times worse), 49 us for one at
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
        const int64_t a = box_elem(m.box, origin, e);
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
        constexpr int KS = KU % 4 == 0 ? 4 : 2;
#pragma unroll 1
        for (int k0 = 0; k0 < NV; k0 += KU) {
            typename P::QP w[KU];
#pragma unroll
            for (int k = 0; k < KU; ++k)
                w[k] = *reinterpret_cast<const typename P::QP *>(Q + (int64_t)(k0 + k) * m.nelem + a);
            // KS rows' products first, then the running sum: it rounds once per KS rows
#pragma unroll
            for (int k = 0; k < KU; k += KS) {
                C<R> q[KS][EPP];
#pragma unroll
                for (int j = 0; j < KS; ++j) P::q(w[k + j], q[j]);
#pragma unroll
                for (int r = 0; r < NB; ++r)
#pragma unroll
                    for (int x = 0; x < EPP; ++x) {
                        C<R> t = mk<R>(0, 0);
#pragma unroll
                        for (int j = 0; j < KS; ++j) cfma(t, q[j][x], cs[k0 + k + j][r]);
                        v[r][x] = v[r][x] + t;
                    }
            }
        }
#pragma unroll
        for (int r = 0; r < NB; ++r)
            if (r < nr) *reinterpret_cast<typename P::FP *>(f + (int64_t)r * m.nelem + a) = piece(v[r]);
    }
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

template void restrict_<double>(dwf_ctx *, const Level &, double2 *, const double2 *, const double2 *);
template void restrict_<float>(dwf_ctx *, const Level &, float2 *, const float2 *, const float2 *);
template void prolong_<double>(dwf_ctx *, const Level &, double2 *, const double2 *, const double2 *, bool);
template void prolong_<float>(dwf_ctx *, const Level &, float2 *, const float2 *, const float2 *, bool);

}  // namespace dwf
