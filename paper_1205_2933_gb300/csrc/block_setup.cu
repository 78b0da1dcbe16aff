// Kernels that build the coarse space (Sec. 2): the Gamma split of the adaptive
// vectors, block Gram matrices, the block Gram-Schmidt as two Cholesky QR
// passes, and the block-face products of the Galerkin operator.
#include <cooperative_groups.h>

#include "blockmap.cuh"

namespace dwf {

namespace cg = cooperative_groups;

namespace {

// How a Gram CTA shares the NV x NV products: a thread keeps GT x GT of them
// (rows and columns GP apart), GSZ threads cover the matrix, EG such groups
// take 16 elements each of a stage.
template <typename R, int NV, bool SAME> struct GShape {
    static constexpr int GT = NV == 32 ? 4 : NV % 3 == 0 ? 3 : 2;
    static constexpr int GP = NV / GT, GSZ = GP * GP;
    static constexpr int EG = GSZ == 1 ? 64 : 256 / GSZ < 16 ? 256 / GSZ : 16;
    static constexpr int NT = GSZ * EG;
    static constexpr int EPP = sizeof(R) == 4 ? 2 : 1;      // elements per 16 bytes
    static constexpr int CH = 16 * EG;                      // elements of one stage
    static constexpr int ROW = CH + EPP;                    // padded: rows start 4 banks apart
    static constexpr size_t stage = sizeof(C<R>) * NV * ROW * (SAME ? 1 : 2);
    static constexpr int NS = 96 * 1024 / stage >= 3 ? 3 : 2;
    static constexpr size_t red = sizeof(double2) * (EG + 1) * NV * NV;
    static constexpr size_t smem = stage * NS > red ? stage * NS : red;
};

// hi + lo += s for FP32 partial sums: Knuth's two-sum keeps what the addition
// rounds off, so that the pair carries about 48 bits (six FP32 additions; an
// FP64 addition and the conversion cost this chip's FP32 pipe 128 of them)
struct Sum2 {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float s) {
        const float t = hi + s, b = t - hi;
        lo += (hi - (t - b)) + (s - b);
        hi = t;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};
struct Sum1 {
    double hi = 0.0;
    __device__ __forceinline__ void add(double s) { hi += s; }
    __device__ __forceinline__ double value() const { return hi; }
};

// G[xc * gld][k][l] = sum over the box of block xc of conj(A_k) B_l.  The box
// starts `off` sites after the block's first site; with `dense` B holds only
// the boxes, one after another.  SAME: B is A.  A cluster of CTAs shares one
// block; every CTA streams its part of the elements through NS stages of
// asynchronous copies, and the cluster's first CTA adds the parts in a fixed
// order.  Sums: 16 products at a time in the field precision, these in FP64 or
// (FP32 fields) as unevaluated pairs, the parts of threads and CTAs in FP64.
// Bound: the FMA pipe of the field precision.  FP64 additions of the 16-product
// sums took 1.90 ms where the pairs take 0.70.
// Nvec 24 on 12^3 x 16 x 16 (FP32): 0.70 ms for Q^+ Q, 16.7 ms with one CTA per
// block, chunks of 16 elements and one product per thread and load pair.
template <typename R, int NV, bool SAME>
__global__ void __launch_bounds__(GShape<R, NV, SAME>::NT)
gram_kernel(double2 *__restrict__ G, int gld, const C<R> *__restrict__ A, const C<R> *__restrict__ B, int64_t bstride,
            int dense, BlockMap m, Box box, int64_t off, unsigned ne) {
    using S = GShape<R, NV, SAME>;
    using V4 = typename std::conditional<sizeof(R) == 4, float4, double2>::type;
    constexpr int GT = S::GT, GP = S::GP, EPP = S::EPP, CH = S::CH, ROW = S::ROW, NS = S::NS, NP = NV * NV;
    constexpr int PIECES = CH / EPP, PT = PIECES < S::NT ? PIECES : S::NT, RS = S::NT / PT;
    extern __shared__ __align__(16) unsigned char smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned cs = cluster.num_blocks(), rank = cluster.block_rank();
    const int64_t xc = blockIdx.x / cs;
    const unsigned nst = (ne + CH - 1) / CH, spc = (nst + cs - 1) / cs;
    const unsigned st0 = rank * spc, st1 = min(nst, st0 + spc);
    const int64_t origin = block_origin(m, xc) + off;
    auto sA = [&](unsigned st) { return reinterpret_cast<C<R> *>(smem + S::stage * (st % NS)); };
    auto fill = [&](unsigned st) {
        if (st < st1) {
            C<R> *a = sA(st), *b = a + NV * ROW;
            for (int p = threadIdx.x % PT; p < PIECES; p += PT) {
                const unsigned e = st * CH + p * EPP;
                const bool in = e < ne;
                const int64_t ad = in ? box_elem(box, origin, e) : 0;
                const int64_t bd = !in ? 0 : dense ? xc * ne + e : ad;
                for (int row = threadIdx.x / PT; row < NV; row += RS) {
                    cp_async<16>(a + row * ROW + p * EPP, A + (int64_t)row * m.nelem + ad, in);
                    if (!SAME) cp_async<16>(b + row * ROW + p * EPP, B + (int64_t)row * bstride + bd, in);
                }
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    const int t = threadIdx.x % S::GSZ, eg = threadIdx.x / S::GSZ;
    const int ka = t / GP, lb = t % GP;
    using Sum = typename std::conditional<sizeof(R) == 4, Sum2, Sum1>::type;
    Sum sre[GT][GT], sim[GT][GT];
#pragma unroll
    for (int i = 0; i < NS - 1; ++i) fill(st0 + i);
    for (unsigned st = st0; st < st1; ++st) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(NS - 2) : "memory");
        __syncthreads();
        fill(st + NS - 1);
        const C<R> *a = sA(st) + ka * ROW + eg * 16;
        const C<R> *b = sA(st) + (SAME ? 0 : NV * ROW) + lb * ROW + eg * 16;
        C<R> s[GT][GT];
#pragma unroll
        for (int i = 0; i < GT; ++i)
#pragma unroll
            for (int j = 0; j < GT; ++j) s[i][j] = mk<R>(0, 0);
#pragma unroll 4
        for (int x = 0; x < 16; x += EPP) {
            V4 av[GT], bv[GT];
#pragma unroll
            for (int i = 0; i < GT; ++i) {
                av[i] = *reinterpret_cast<const V4 *>(a + i * GP * ROW + x);
                bv[i] = *reinterpret_cast<const V4 *>(b + i * GP * ROW + x);
            }
#pragma unroll
            for (int i = 0; i < GT; ++i)
#pragma unroll
                for (int j = 0; j < GT; ++j) {
                    cfmac(s[i][j], mk<R>(av[i].x, av[i].y), mk<R>(bv[j].x, bv[j].y));
                    if constexpr (EPP == 2) cfmac(s[i][j], mk<R>(av[i].z, av[i].w), mk<R>(bv[j].z, bv[j].w));
                }
        }
#pragma unroll
        for (int i = 0; i < GT; ++i)
#pragma unroll
            for (int j = 0; j < GT; ++j) {
                sre[i][j].add(s[i][j].x);
                sim[i][j].add(s[i][j].y);
            }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    double2 *red = reinterpret_cast<double2 *>(smem), *mine = red + S::EG * NP;
#pragma unroll
    for (int i = 0; i < GT; ++i)
#pragma unroll
        for (int j = 0; j < GT; ++j)
            red[eg * NP + (ka + i * GP) * NV + lb + j * GP] = make_double2(sre[i][j].value(), sim[i][j].value());
    __syncthreads();
    for (int p = threadIdx.x; p < NP; p += S::NT) {
        double2 v = red[p];
#pragma unroll 4
        for (int h = 1; h < S::EG; ++h) v = v + red[h * NP + p];
        mine[p] = v;
    }
    cluster.sync();
    if (rank == 0)
        for (int p = threadIdx.x; p < NP; p += S::NT) {
            double2 v = mine[p];
            for (unsigned h = 1; h < cs; ++h) v = v + cluster.map_shared_rank(mine, h)[p];
            G[xc * gld * NP + p] = v;
        }
    cluster.sync();  // the parts stay readable until the first CTA has added them
}

template <typename R, int NV, bool SAME>
void gram_launch(dwf_ctx *c, double2 *G, int gld, const C<R> *A, const C<R> *B, int64_t bstride, bool dense,
                 const BlockMap &m, const Box &box, int64_t off, int64_t ne) {
    using S = GShape<R, NV, SAME>;
    auto *fn = gram_kernel<R, NV, SAME>;
    const int64_t nc = ncoarse(m), stages = (ne + S::CH - 1) / S::CH;
    int cs = 1;
    while (cs < 8 && nc * cs < 2 * (int64_t)c->sm_count && stages >= 4 * cs) cs *= 2;
    DWF_REQUIRE(nc * cs < ((int64_t)1 << 31) && ne < ((int64_t)1 << 30), DWF_EINVAL, "block Gram grid too large");
    if (S::smem > 48 * 1024)
        DWF_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem));
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)cs;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(nc * cs));
    cfg.blockDim = dim3(S::NT);
    cfg.dynamicSmemBytes = S::smem;
    cfg.stream = c->stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    DWF_CUDA(cudaLaunchKernelEx(&cfg, fn, G, gld, A, B, bstride, dense ? 1 : 0, m, box, off, (unsigned)ne));
    DWF_CHECK_LAUNCH();
}

// Cholesky G = R^+ R (R upper triangular, positive diagonal) and Rinv = R^-1
// in FP64, one CTA per coarse site, the matrix in shared memory: row j is
// scaled, then subtracted from the rows below it by all threads; the inverse
// row by row from the last one up, one column per thread.  *bad gets 1 where
// a pivot is lost.  Bound by its chain of 2 Nvec dependent steps: below 0.1 ms at
// Nvec 24, where one thread per site took 1.6 ms.
__global__ void __launch_bounds__(256) chol_inv_kernel(const double2 *__restrict__ G, double2 *__restrict__ Ri, int *bad,
                                                       int nv) {
    extern __shared__ __align__(16) unsigned char smem[];
    double2 *r = reinterpret_cast<double2 *>(smem);  // [nv][nv]: G, then R in its upper triangle
    double2 *x = r + nv * nv;                        // [nv][nv]: R^-1
    __shared__ double g0[32];                        // the diagonal of G
    const double2 *g = G + (int64_t)blockIdx.x * nv * nv;
    for (int i = threadIdx.x; i < nv * nv; i += blockDim.x) {
        r[i] = g[i];
        x[i] = make_double2(0, 0);
    }
    if (threadIdx.x < nv) g0[threadIdx.x] = g[threadIdx.x * nv + threadIdx.x].x;
    __syncthreads();
    for (int j = 0; j < nv; ++j) {
        const double d = r[j * nv + j].x;
        if (!(d > 1e-28 * fabs(g0[j])) || !(d > 0.0)) {  // the same for every thread
            if (threadIdx.x == 0) atomicExch(bad, 1);
            return;
        }
        const double rd = sqrt(d);
        __syncthreads();  // everyone has read the pivot
        if (threadIdx.x == j) r[j * nv + j] = make_double2(rd, 0);
        else if (threadIdx.x > j && threadIdx.x < nv) {
            const double2 v = r[j * nv + threadIdx.x];
            r[j * nv + threadIdx.x] = make_double2(v.x / rd, v.y / rd);
        }
        __syncthreads();
        const int left = nv - 1 - j;
        for (int p = threadIdx.x; p < left * left; p += blockDim.x) {
            const int i = j + 1 + p / left, k = j + 1 + p % left;
            if (k < i) continue;
            const double2 t = cmulc(r[j * nv + i], r[j * nv + k]);
            r[i * nv + k].x -= t.x;
            r[i * nv + k].y -= t.y;
        }
        __syncthreads();
    }
    // R X = 1 with X upper triangular
    for (int i = nv - 1; i >= 0; --i) {
        const int col = threadIdx.x;
        if (col >= i && col < nv) {
            double2 s = make_double2(i == col ? 1.0 : 0.0, 0.0);
            for (int k = i + 1; k <= col; ++k) {
                const double2 t = cmul(r[i * nv + k], x[k * nv + col]);
                s.x -= t.x;
                s.y -= t.y;
            }
            const double dinv = 1.0 / r[i * nv + i].x;
            x[i * nv + col] = make_double2(s.x * dinv, s.y * dinv);
        }
    }
    __syncthreads();
    double2 *ri = Ri + (int64_t)blockIdx.x * nv * nv;
    for (int i = threadIdx.x; i < nv * nv; i += blockDim.x) ri[i] = x[i];
}

// Q_l <- sum_{k <= l} Q_k Rinv[k][l] in place.  grid.x = coarse sites x pieces
// of a block; a thread takes 16 bytes of every basis row and forms LG rows at
// a time, the last ones first (they read rows that are still the old ones),
// from coefficients in shared memory.  Holding all rows in registers instead
// spilled.  Bound by reading and writing the basis (the repeated reads hit
// L1/L2): Nvec 24 on 12^3 x 16 x 16 (FP32, 2.0 GB) 0.43 ms
// (one CTA per block: 5.4 ms)
constexpr int AT = 128;
template <typename R, int NV>
__global__ void __launch_bounds__(AT) apply_rinv_kernel(C<R> *__restrict__ Q, const double2 *__restrict__ Ri, BlockMap m,
                                                        int pieces) {
    constexpr int EPP = sizeof(R) == 4 ? 2 : 1, LG = NV % 8 == 0 ? 8 : NV % 6 == 0 ? 6 : NV;
    struct alignas(16) Vec {
        C<R> e[EPP];
    };
    __shared__ __align__(16) C<R> r[NV * NV];
    const int64_t xc = blockIdx.x / pieces;
    const unsigned part = blockIdx.x - (unsigned)xc * pieces;
    for (int i = threadIdx.x; i < NV * NV; i += AT) r[i] = cvt<C<R>, double2>(Ri[xc * NV * NV + i]);
    __syncthreads();
    const unsigned ne = (unsigned)(m.bsites * m.run);
    const int64_t origin = block_origin(m, xc);
    for (unsigned e = (part * AT + threadIdx.x) * EPP; e < ne; e += (unsigned)pieces * AT * EPP) {
        C<R> *q = Q + box_elem(m.box, origin, e);
#pragma unroll 1
        for (int l0 = NV - LG; l0 >= 0; l0 -= LG) {
            Vec s[LG];
#pragma unroll
            for (int l = 0; l < LG; ++l)
#pragma unroll
                for (int x = 0; x < EPP; ++x) s[l].e[x] = mk<R>(0, 0);
#pragma unroll 4
            for (int k = 0; k < l0 + LG; ++k) {  // Rinv[k][l] = 0 for k > l
                const Vec v = *reinterpret_cast<const Vec *>(q + k * m.nelem);
#pragma unroll
                for (int l = 0; l < LG; ++l)
#pragma unroll
                    for (int x = 0; x < EPP; ++x) cfma(s[l].e[x], v.e[x], r[k * NV + l0 + l]);
            }
#pragma unroll
            for (int l = 0; l < LG; ++l) *reinterpret_cast<Vec *>(q + (l0 + l) * m.nelem) = s[l];
        }
    }
}

// Gamma split of adaptive vectors into Q (see mg.cuh).  The halving follows
// the conversion (exact), so that FP64 spends one addition per real part.
template <typename R>
__global__ void __launch_bounds__(256) gamma_split_kernel(C<R> *__restrict__ Q, const double2 *__restrict__ v, int nadapt,
                                                          int split, int64_t nelem, int ncomp, int Ls, int fine) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nelem; i += (int64_t)gridDim.x * blockDim.x) {
        const int s = (int)(i % Ls);
        const int comp = (int)(i / Ls % ncomp);
        const int64_t refl = i + Ls - 1 - 2 * s;  // the element at Ls - 1 - s
        // Gamma on the fine level: gamma_5 (sign of comp) and the reflection of
        // s; on a coarse level the sign of even and odd components
        const bool neg = fine ? comp >= 6 : (comp & 1);
#pragma unroll 4
        for (int j = 0; j < nadapt; ++j) {
            const double2 a = v[j * nelem + i];
            if (!split) {
                Q[j * nelem + i] = cvt<C<R>, double2>(a);
                continue;
            }
            const double2 b = fine ? v[j * nelem + refl] : a;
            const double2 p = a + b, n = a - b;
            const C<R> hp = mk<R>(R(0.5) * (R)p.x, R(0.5) * (R)p.y), hn = mk<R>(R(0.5) * (R)n.x, R(0.5) * (R)n.y);
            Q[(2 * j) * nelem + i] = neg ? hn : hp;
            Q[(2 * j + 1) * nelem + i] = neg ? hp : hn;
        }
    }
}

}  // namespace

template <typename R> void block_gram(dwf_ctx *c, const Level &L, double2 *G, const C<R> *A, const C<R> *B) {
    const BlockMap m = make_map(L);
#define GK(NV)                                                                                                        \
    if (A == B) gram_launch<R, NV, true>(c, G, 1, A, A, m.nelem, false, m, m.box, 0, m.bsites * m.run);               \
    else gram_launch<R, NV, false>(c, G, 1, A, B, m.nelem, false, m, m.box, 0, m.bsites * m.run)
    NV_DISPATCH(L.nv, GK);
#undef GK
}

template <typename R>
void face_gram(dwf_ctx *c, const Level &L, double2 *F, const C<R> *Q, const C<R> *H, int64_t hstride, int mu, int dir) {
    const BlockMap m = make_map(L);
    int n[4] = {m.b[0], m.b[1], m.b[2], m.b[3]};
    n[mu] = 1;
    const Box box = make_box(n, m.L, m.run);
    int64_t off = dir > 0 ? m.b[mu] - 1 : 0;
    for (int i = 0; i < mu; ++i) off *= m.L[i];
    const int dd = 2 * mu + (dir > 0 ? 0 : 1);
#define GK(NV) \
    gram_launch<R, NV, false>(c, F + (size_t)dd * NV * NV, 8, Q, H, hstride, true, m, box, off, m.bsites / m.b[mu] * m.run)
    NV_DISPATCH(L.nv, GK);
#undef GK
}

template <typename R> bool block_orthonormalise(dwf_ctx *c, Level &L, C<R> *Q) {
    const BlockMap m = make_map(L);
    const int64_t nc = ncoarse(m), ne = m.bsites * m.run;
    const size_t gb = sizeof(double2) * nc * L.nv * L.nv;
    if (L.G.bytes < gb) L.G.alloc(gb);
    if (L.Rinv.bytes < gb) L.Rinv.alloc(gb);
    if (L.info.bytes < sizeof(int)) L.info.alloc(sizeof(int));
    DWF_CUDA(cudaMemsetAsync(L.info.p, 0, sizeof(int), c->stream));
    for (int pass = 0; pass < 2; ++pass) {  // CholQR2
        block_gram<R>(c, L, L.G.as<double2>(), Q, Q);
        chol_inv_kernel<<<(unsigned)nc, 256, 2 * sizeof(double2) * L.nv * L.nv, c->stream>>>(
            L.G.as<double2>(), L.Rinv.as<double2>(), L.info.as<int>(), L.nv);
        DWF_CHECK_LAUNCH();
#define AK(NV)                                                                                                      \
    {                                                                                                               \
        constexpr int EPP = sizeof(R) == 4 ? 2 : 1;                                                                 \
        const int64_t one = (ne + AT * EPP - 1) / (AT * EPP);                                                       \
        const int pieces = (int)std::min<int64_t>(one, std::max<int64_t>(1, (32 * (int64_t)c->sm_count + nc - 1) / nc)); \
        apply_rinv_kernel<R, NV><<<(unsigned)(nc * pieces), AT, 0, c->stream>>>(Q, L.Rinv.as<double2>(), m, pieces); \
    }
        NV_DISPATCH(L.nv, AK);
#undef AK
        DWF_CHECK_LAUNCH();
    }
    int bad = 0;  // a lost pivot in either pass (the basis is then discarded)
    DWF_CUDA(cudaMemcpyAsync(&bad, L.info.p, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    DWF_CUDA(cudaStreamSynchronize(c->stream));
    return bad == 0;
}

template <typename R> void gamma_split(dwf_ctx *c, const Level &L, C<R> *Q, const double2 *v, int nadapt, bool split) {
    int64_t n = L.lg.nelem;
    unsigned blocks = (unsigned)std::min<int64_t>((n + 255) / 256, (int64_t)c->sm_count * 16);
    gamma_split_kernel<R><<<blocks, 256, 0, c->stream>>>(Q, v, nadapt, split ? 1 : 0, n, L.lg.ncomp, L.lg.g.Ls,
                                                         L.index == 0 ? 1 : 0);
    DWF_CHECK_LAUNCH();
}

template void block_gram<double>(dwf_ctx *, const Level &, double2 *, const double2 *, const double2 *);
template void block_gram<float>(dwf_ctx *, const Level &, double2 *, const float2 *, const float2 *);
template void face_gram<double>(dwf_ctx *, const Level &, double2 *, const double2 *, const double2 *, int64_t, int, int);
template void face_gram<float>(dwf_ctx *, const Level &, double2 *, const float2 *, const float2 *, int64_t, int, int);
template bool block_orthonormalise<double>(dwf_ctx *, Level &, double2 *);
template bool block_orthonormalise<float>(dwf_ctx *, Level &, float2 *);
template void gamma_split<double>(dwf_ctx *, const Level &, double2 *, const double2 *, int, bool);
template void gamma_split<float>(dwf_ctx *, const Level &, float2 *, const double2 *, int, bool);

}  // namespace dwf
