// Level-1 vector kernels.  Reductions accumulate in FP64 whatever the
// storage precision and are deterministic: every CTA writes a partial sum,
// and the last CTA to finish (atomic ticket) adds the partials in a fixed
// order and stores the result in a device scalar slot, so that solver
// coefficients can stay on the GPU.
#include "reduce.cuh"

namespace dwf {

namespace {

constexpr int RED_THREADS = 256;
constexpr int RED_MAX_BLOCKS = 1024;

// Per-thread partial sums in the storage precision (FP32 FMAs for FP32
// fields), combined across threads and CTAs in FP64.  Fused multiply-adds, one
// product each (the FP64 pipe bounds these loops), in two chains per sum: each
// rounds at half the size of the whole, so that both together round no worse
// than one chain of two products at a time.
template <typename T> struct Acc;
template <> struct Acc<double2> { using type = double; };
template <> struct Acc<float2> { using type = float; };

template <typename TX, typename TY>
__global__ void __launch_bounds__(RED_THREADS) dot_kernel(const TX *__restrict__ x, const TY *__restrict__ y, int64_t n,
                                                          double *part, unsigned *count, double *out) {
    using A = typename Acc<TX>::type;
    A ar[2] = {0, 0}, ai[2] = {0, 0};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        TX u = x[i];
        TY v = y[i];
        ar[0] += (A)u.x * (A)v.x;
        ai[0] += (A)u.x * (A)v.y;
        ar[1] += (A)u.y * (A)v.y;
        ai[1] -= (A)u.y * (A)v.x;
    }
    const double m[2] = {(double)(ar[0] + ar[1]), (double)(ai[0] + ai[1])};
    grid_sums<2>(m, part, count, out, 2);
}

template <typename T>
__global__ void __launch_bounds__(RED_THREADS) norm2_kernel(const T *__restrict__ x, int64_t n, double *part,
                                                            unsigned *count, double *out) {
    using A = typename Acc<T>::type;
    A a[2] = {0, 0};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        T u = x[i];
        a[0] += (A)u.x * (A)u.x;
        a[1] += (A)u.y * (A)u.y;
    }
    const double m[1] = {(double)(a[0] + a[1])};
    grid_sums<1>(m, part, count, out, 1);
}

// out[2j], out[2j+1] = <V_j, w> for j < K: w is read once for K vectors.
template <typename T, int K> struct MultiDotArgs {
    const T *v[K];
};

template <typename T, int K>
__global__ void __launch_bounds__(RED_THREADS) multidot_kernel(MultiDotArgs<T, K> a, const T *__restrict__ w, int64_t n,
                                                               double *part, unsigned *count, double *out) {
    using A = typename Acc<T>::type;
    A ar[K][2], ai[K][2];
#pragma unroll
    for (int j = 0; j < K; ++j) ar[j][0] = ar[j][1] = ai[j][0] = ai[j][1] = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        T y = w[i];
#pragma unroll
        for (int j = 0; j < K; ++j) {
            T u = a.v[j][i];
            ar[j][0] += (A)u.x * (A)y.x;
            ai[j][0] += (A)u.x * (A)y.y;
            ar[j][1] += (A)u.y * (A)y.y;
            ai[j][1] -= (A)u.y * (A)y.x;
        }
    }
    double m[2 * K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        m[2 * j] = (double)(ar[j][0] + ar[j][1]);
        m[2 * j + 1] = (double)(ai[j][0] + ai[j][1]);
    }
    grid_sums<2 * K>(m, part, count, out, 2 * K);
}

template <typename T>
__global__ void zero_kernel(T *x, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        x[i] = cvt<T, double2>(make_double2(0, 0));
}

template <typename TO, typename TI>
__global__ void copy_kernel(TO *__restrict__ out, const TI *__restrict__ in, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = cvt<TO, TI>(in[i]);
}

// at least four elements per thread: every CTA ends with a ticket on one address
unsigned red_blocks(dwf_ctx *c, int64_t n) {
    int64_t b = std::max<int64_t>((n + 4 * RED_THREADS - 1) / (4 * RED_THREADS),
                                  std::min<int64_t>((n + RED_THREADS - 1) / RED_THREADS, c->sm_count));
    int64_t cap = std::min<int64_t>(RED_MAX_BLOCKS, (int64_t)c->sm_count * 6);
    return (unsigned)std::max<int64_t>(1, std::min(b, cap));
}

unsigned ew_blocks(dwf_ctx *c, int64_t n) {
    int64_t b = (n + 255) / 256;
    int64_t cap = (int64_t)c->sm_count * 16;
    return (unsigned)std::max<int64_t>(1, std::min(b, cap));
}

}  // namespace

template <typename T> void bzero(dwf_ctx *c, T *x, int64_t n) {
    zero_kernel<T><<<ew_blocks(c, n), 256, 0, c->stream>>>(x, n);
    DWF_CHECK_LAUNCH();
}

template <typename TO, typename TI> void bcopy(dwf_ctx *c, TO *out, const TI *in, int64_t n) {
    copy_kernel<TO, TI><<<ew_blocks(c, n), 256, 0, c->stream>>>(out, in, n);
    DWF_CHECK_LAUNCH();
}

template <typename TX, typename TY> void bdot(dwf_ctx *c, int slot, const TX *x, const TY *y, int64_t n) {
    dot_kernel<TX, TY><<<red_blocks(c, n), RED_THREADS, 0, c->stream>>>(
        x, y, n, c->red_part.as<double>(), c->red_count.as<unsigned>(), c->scal.as<double>() + slot);
    DWF_CHECK_LAUNCH();
}

template <typename T> void bnorm2(dwf_ctx *c, int slot, const T *x, int64_t n) {
    norm2_kernel<T><<<red_blocks(c, n), RED_THREADS, 0, c->stream>>>(
        x, n, c->red_part.as<double>(), c->red_count.as<unsigned>(), c->scal.as<double>() + slot);
    DWF_CHECK_LAUNCH();
}

static unsigned long long g_launches = 0;
void note_launch() { __atomic_add_fetch(&g_launches, 1ull, __ATOMIC_RELAXED); }
void note_launches(unsigned long long n) { __atomic_add_fetch(&g_launches, n, __ATOMIC_RELAXED); }
unsigned long long launch_count() { return __atomic_load_n(&g_launches, __ATOMIC_RELAXED); }

static cudaEvent_t take_event(dwf_ctx *c) {
    if (!c->prof_pool.empty()) {
        cudaEvent_t e = c->prof_pool.back();
        c->prof_pool.pop_back();
        return e;
    }
    cudaEvent_t e;
    DWF_CUDA(cudaEventCreate(&e));
    return e;
}

// Inside a graph capture the events are recorded as event-record nodes of
// the graph (cudaEventRecordExternal), so that every replay records them.
static cudaError_t record(dwf_ctx *c, cudaEvent_t e) {
    return c->cap_rec ? cudaEventRecordWithFlags(e, c->stream, cudaEventRecordExternal) : cudaEventRecord(e, c->stream);
}

ProfScope::ProfScope(dwf_ctx *ctx, int k, int nunits) : c(ctx), cls(k), units(nunits) {
    if (!c->prof) return;
    a = take_event(c);
    b = take_event(c);
    DWF_CUDA(record(c, a));
}

ProfScope::~ProfScope() {
    if (!a) return;
    if (record(c, b) == cudaSuccess)
        (c->cap_rec ? *c->cap_rec : c->prof_rec).push_back(ProfRecord{cls, a, b, units, -1.f});
}

void prof_reset(dwf_ctx *c) {
    for (auto &r : c->prof_rec)
        if (r.a) {
            c->prof_pool.push_back(r.a);
            c->prof_pool.push_back(r.b);
        }
    c->prof_rec.clear();
}

template <typename T> void bmultidot(dwf_ctx *c, int slot, T *const *V, int k, const T *w, int64_t n) {
    for (int j0 = 0; j0 < k; j0 += 8) {
        int kk = std::min(8, k - j0);
        unsigned nb = red_blocks(c, n);
#define MD(K)                                                                                            \
    {                                                                                                    \
        MultiDotArgs<T, K> a;                                                                            \
        for (int j = 0; j < K; ++j) a.v[j] = V[j0 + j];                                                  \
        multidot_kernel<T, K><<<nb, RED_THREADS, 0, c->stream>>>(a, w, n, c->red_part.as<double>(),     \
                                                                 c->red_count.as<unsigned>(),            \
                                                                 c->scal.as<double>() + slot + 2 * j0);  \
    }
        switch (kk) {
            case 1: MD(1) break;
            case 2: MD(2) break;
            case 3: MD(3) break;
            case 4: MD(4) break;
            case 5: MD(5) break;
            case 6: MD(6) break;
            case 7: MD(7) break;
            default: MD(8) break;
        }
#undef MD
        DWF_CHECK_LAUNCH();
    }
}

double read_scalar(dwf_ctx *c, int slot) {
    double v;
    read_scalars(c, slot, 1, &v);
    return v;
}

void read_scalars(dwf_ctx *c, int slot, int count, double *out) {
    DWF_CUDA(cudaMemcpyAsync(c->hscal, c->scal.as<double>() + slot, sizeof(double) * count,
                             cudaMemcpyDeviceToHost, c->stream));
    DWF_CUDA(cudaStreamSynchronize(c->stream));
    for (int i = 0; i < count; ++i) out[i] = c->hscal[i];
}

void write_scalar(dwf_ctx *c, int slot, double v) {
    DWF_CUDA(cudaMemcpyAsync(c->scal.as<double>() + slot, &v, sizeof(double), cudaMemcpyHostToDevice, c->stream));
    DWF_CUDA(cudaStreamSynchronize(c->stream));
}

#define INST2(TX, TY) template void bdot<TX, TY>(dwf_ctx *, int, const TX *, const TY *, int64_t); \
                      template void bcopy<TX, TY>(dwf_ctx *, TX *, const TY *, int64_t);
INST2(double2, double2)
INST2(double2, float2)
INST2(float2, double2)
INST2(float2, float2)
template void bzero<double2>(dwf_ctx *, double2 *, int64_t);
template void bzero<float2>(dwf_ctx *, float2 *, int64_t);
template void bnorm2<double2>(dwf_ctx *, int, const double2 *, int64_t);
template void bmultidot<double2>(dwf_ctx *, int, double2 *const *, int, const double2 *, int64_t);
template void bmultidot<float2>(dwf_ctx *, int, float2 *const *, int, const float2 *, int64_t);
template void bnorm2<float2>(dwf_ctx *, int, const float2 *, int64_t);

}  // namespace dwf
