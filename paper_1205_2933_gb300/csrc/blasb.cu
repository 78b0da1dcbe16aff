// Batched vector kernels: nrhs fields of n elements stored one after the
// other, blockIdx.y = right-hand side.  Every right-hand side has its own
// coefficients, read from device memory (scalar slots or coefficient
// arrays), and its own deterministic FP64-accumulated reductions.
#include "mg.cuh"
#include "reduce.cuh"

namespace dwf {

namespace {

constexpr int BT = 256;

template <typename T> struct RealB;
template <> struct RealB<float2> { using type = float; };
template <> struct RealB<double2> { using type = double; };

// Sums are kept in several chains, one per part of a product or more: a thread
// adds up more elements than when every element had a CTA's share to itself, and
// shorter chains at a fraction of the sum's size round no worse.
// s[base + r*stride] = |x_r|^2
template <typename T>
__global__ void __launch_bounds__(BT) norm2_b_kernel(const T *__restrict__ x, int64_t n, double *part, unsigned *count,
                                                     double *s, int base, int stride) {
    using A = typename RealB<T>::type;
    x += (size_t)blockIdx.y * n;
    A a[2][2] = {{0, 0}, {0, 0}};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n / Pack<T>::N; i += (int64_t)gridDim.x * blockDim.x) {
        const Pack<T> u = ldp(x, i);
#pragma unroll
        for (int e = 0; e < Pack<T>::N; ++e) {
            a[e][0] += u.e[e].x * u.e[e].x;
            a[e][1] += u.e[e].y * u.e[e].y;
        }
    }
    const double m[1] = {(double)((a[0][0] + a[0][1]) + (a[1][0] + a[1][1]))};
    grid_sums<1>(m, part + (size_t)blockIdx.y * gridDim.x, count + blockIdx.y, s + base + blockIdx.y * stride, 1);
}

// s[base + r*stride + 2j (+1)] = <V_j,r, w_r>, j < K (w read once)
template <typename T, int K> struct VArgs {
    const T *v[K];
};
template <typename T, int K>
__global__ void __launch_bounds__(BT) multidot_b_kernel(VArgs<T, K> va, const T *__restrict__ w, int64_t n,
                                                        double *part, unsigned *count, double *s, int base,
                                                        int stride) {
    using A = typename RealB<T>::type;
    const size_t off = (size_t)blockIdx.y * n;
    A ar[K][2], ai[K][2];
#pragma unroll
    for (int j = 0; j < K; ++j) ar[j][0] = ar[j][1] = ai[j][0] = ai[j][1] = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n / Pack<T>::N; i += (int64_t)gridDim.x * blockDim.x) {
        const Pack<T> y = ldp(w + off, i);
        Pack<T> u[K];
#pragma unroll
        for (int j = 0; j < K; ++j) u[j] = ldp(va.v[j] + off, i);
#pragma unroll
        for (int j = 0; j < K; ++j)
#pragma unroll
            for (int e = 0; e < Pack<T>::N; ++e) {
                ar[j][0] += u[j].e[e].x * y.e[e].x;
                ai[j][0] += u[j].e[e].x * y.e[e].y;
                ar[j][1] += u[j].e[e].y * y.e[e].y;
                ai[j][1] -= u[j].e[e].y * y.e[e].x;
            }
    }
    double m[2 * K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
        m[2 * j] = (double)(ar[j][0] + ar[j][1]);
        m[2 * j + 1] = (double)(ai[j][0] + ai[j][1]);
    }
    grid_sums<2 * K>(m, part + (size_t)blockIdx.y * 2 * K * gridDim.x, count + blockIdx.y,
                     s + base + blockIdx.y * stride, 2 * K);
}

// w_r += sgn * sum_j c_{r,j} V_j,r with c from slots s[base + r*stride + 2j]
template <typename T> struct MArgs {
    const T *v[32];
    int k;
};
template <typename T>
__global__ void multiaxpy_b_kernel(T *__restrict__ w, MArgs<T> a, const double *__restrict__ s, int base, int stride,
                                   double sgn, int64_t n) {
    using R = typename RealB<T>::type;
    const int r = blockIdx.y;
    const size_t off = (size_t)r * n;
    __shared__ R cr[32], ci[32];  // (indexed registers would live in local memory)
    if (threadIdx.x < a.k) {
        cr[threadIdx.x] = (R)(sgn * s[base + r * stride + 2 * threadIdx.x]);
        ci[threadIdx.x] = (R)(sgn * s[base + r * stride + 2 * threadIdx.x + 1]);
    }
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n / Pack<T>::N; i += (int64_t)gridDim.x * blockDim.x) {
        Pack<T> v = ldp<T>(w + off, i), t{};
#pragma unroll 8
        for (int j = 0; j < a.k; ++j) {
            const Pack<T> u = ldp(a.v[j] + off, i);
#pragma unroll
            for (int e = 0; e < Pack<T>::N; ++e) {
                t.e[e].x += cr[j] * u.e[e].x;  // small against v, which is rounded once
                t.e[e].y += cr[j] * u.e[e].y;
                t.e[e].x -= ci[j] * u.e[e].y;
                t.e[e].y += ci[j] * u.e[e].x;
            }
        }
#pragma unroll
        for (int e = 0; e < Pack<T>::N; ++e) v.e[e] = v.e[e] + t.e[e];
        stp(w + off, i, v);
    }
}

// The CGNR step split so that every field is read once per iteration:
//   r:  a = s[izz] / s[iww]; r -= a w
//   px: a as above, b = s[inew] / s[izz]; x += a p; p = z + b p
//   x:  x += a p (the last iteration, whose residual is not needed)
//   p:  b as above; p' = z + b p
// r and p stand between two Dslash kernels and launch as their dependents
// (launch_after), hence the wait and the plain pointers: a FP32 V-cycle of one
// field of 8^3 x 16 x 16, 15 of each, takes 0.99 ms, with ordinary launches and
// 8-byte accesses 1.14.  Bound by three passes over the field (L2 or DRAM) and
// the launch.
template <typename T>
__global__ void cg_r_b_kernel(T *rout, const T *rin, const T *w, const double *s, int base, int stride, int izz, int iww,
                              int64_t n) {
    using R = typename RealB<T>::type;
    pdl_wait();
    const int r = blockIdx.y;
    const size_t off = (size_t)r * n;
    const double ww = s[base + r * stride + iww];
    const R a = ww > 0.0 ? (R)(s[base + r * stride + izz] / ww) : R(0);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n / Pack<T>::N; i += (int64_t)gridDim.x * blockDim.x) {
        Pack<T> rv = ldp(rin + off, i);
        const Pack<T> wv = ldp(w + off, i);
#pragma unroll
        for (int e = 0; e < Pack<T>::N; ++e) {
            rv.e[e].x -= a * wv.e[e].x;
            rv.e[e].y -= a * wv.e[e].y;
        }
        stp(rout + off, i, rv);
    }
}
template <typename T>
__global__ void cg_p_b_kernel(T *pout, const T *pin, const T *z, const double *s, int base, int stride, int izz, int inew,
                              int64_t n) {
    using R = typename RealB<T>::type;
    pdl_wait();
    const int r = blockIdx.y;
    const size_t off = (size_t)r * n;
    const double zz = s[base + r * stride + izz];
    const R b = zz > 0.0 ? (R)(s[base + r * stride + inew] / zz) : R(0);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n / Pack<T>::N; i += (int64_t)gridDim.x * blockDim.x) {
        Pack<T> pv = ldp(pin + off, i);
        const Pack<T> zv = ldp(z + off, i);
#pragma unroll
        for (int e = 0; e < Pack<T>::N; ++e) {
            pv.e[e].x = zv.e[e].x + b * pv.e[e].x;
            pv.e[e].y = zv.e[e].y + b * pv.e[e].y;
        }
        stp(pout + off, i, pv);
    }
}
template <typename T>
__global__ void cg_px_b_kernel(T *__restrict__ x, T *pout, const T *pin, const T *__restrict__ z,
                               const double *__restrict__ s, int base, int stride, int izz, int iww, int inew,
                               int64_t n, int last, int xinit) {
    using R = typename RealB<T>::type;
    const int r = blockIdx.y;
    const size_t off = (size_t)r * n;
    const double ww = s[base + r * stride + iww], zz = s[base + r * stride + izz];
    const R a = ww > 0.0 ? (R)(zz / ww) : R(0);
    const R b = (!last && zz > 0.0) ? (R)(s[base + r * stride + inew] / zz) : R(0);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        T pv = pin[off + i];
        T xv;
        if (xinit) {
            xv.x = a * pv.x;
            xv.y = a * pv.y;
        } else {
            xv = x[off + i];
            xv.x += a * pv.x;
            xv.y += a * pv.y;
        }
        x[off + i] = xv;
        if (!last) {
            const T zv = z[off + i];
            pv.x = zv.x + b * pv.x;
            pv.y = zv.y + b * pv.y;
            pout[off + i] = pv;
        }
    }
}

// CGNR direction update with the solution update x += a p deferred: up to
// CG_MAXDEFER directions whose steps are not in x yet wait in buffers of
// their own, their steps in the scalar slots ia, ia+1, ...  a = zz/ww and
// b = z'z'/zz of the current iteration as in cg_px_b.
//   mode 0 (defer): pout = z + b pin; s[ia + NP] = a (pin joins the pending)
//   mode 1 (flush): x += sum_j s[ia + j] pend[j] + a pin; pout = z + b pin
//   mode 2 (flush, last iteration): x += sum_j s[ia + j] pend[j] + a pin
// pout may be one of the pending buffers (each element is read before it is written).
template <typename T> struct Pending {
    const T *p[CG_MAXDEFER];
};
template <typename T, int NP>
__global__ void cg_pxd_b_kernel(T *__restrict__ x, T *pout, const T *__restrict__ pin, Pending<T> pend,
                                const T *__restrict__ z, double *s, int base, int stride, int izz, int iww, int inew,
                                int ia, int64_t n, int mode) {
    using R = typename RealB<T>::type;
    const int r = blockIdx.y;
    const size_t off = (size_t)r * n;
    double *sr = s + base + (size_t)r * stride;
    const double ww = sr[iww], zz = sr[izz];
    const R a = ww > 0.0 ? (R)(zz / ww) : R(0);
    const R b = (mode != 2 && zz > 0.0) ? (R)(sr[inew] / zz) : R(0);
    R ap[NP > 0 ? NP : 1];
#pragma unroll
    for (int j = 0; j < NP; ++j) ap[j] = mode != 0 ? (R)sr[ia + j] : R(0);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        T pv = pin[off + i];
        if (mode != 0) {
            T xv = x[off + i];
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const T qv = pend.p[j][off + i];
                xv.x += ap[j] * qv.x;
                xv.y += ap[j] * qv.y;
            }
            xv.x += a * pv.x;
            xv.y += a * pv.y;
            x[off + i] = xv;
        }
        if (mode != 2) {
            const T zv = z[off + i];
            pv.x = zv.x + b * pv.x;
            pv.y = zv.y + b * pv.y;
            pout[off + i] = pv;
        }
    }
    // a defer launch reads no pending step, so no CTA can see this slot change
    if (mode == 0 && blockIdx.x == 0 && threadIdx.x == 0) sr[ia + NP] = (double)a;
}

// out_r = x_r / |x_r| in FP64, |x_r|^2 in s[base + r*stride]
template <typename T>
__global__ void normalised_b_kernel(double2 *__restrict__ out, const T *__restrict__ x, const double *__restrict__ s,
                                    int base, int stride, int64_t n) {
    const size_t off = (size_t)blockIdx.y * n;
    const double a = 1.0 / sqrt(s[base + blockIdx.y * stride]);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const T v = x[off + i];
        out[off + i] = make_double2(a * (double)v.x, a * (double)v.y);
    }
}

// w_r *= scale[r];  res_r -= al[r] * w_r   (GCR direction normalisation and residual update)
template <typename T>
__global__ void gcr_wr_b_kernel(T *__restrict__ w, T *__restrict__ res, GcrStep step, int64_t n) {
    using R = typename RealB<T>::type;
    const int r = blockIdx.y;
    const size_t off = (size_t)r * n;
    const R s = (R)step.scale[r], ar = (R)step.al[r].x, ai = (R)step.al[r].y;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n / Pack<T>::N; i += (int64_t)gridDim.x * blockDim.x) {
        Pack<T> wv = ldp<T>(w + off, i), rv = ldp<T>(res + off, i);
#pragma unroll
        for (int e = 0; e < Pack<T>::N; ++e) {
            wv.e[e].x *= s;
            wv.e[e].y *= s;
            rv.e[e].x -= ar * wv.e[e].x - ai * wv.e[e].y;
            rv.e[e].y -= ar * wv.e[e].y + ai * wv.e[e].x;
        }
        stp(w + off, i, wv);
        stp(res + off, i, rv);
    }
}

// x_r += sum_j g[r*k + j] V_j,r (per-RHS coefficient arrays, k <= 32)
template <typename T>
__global__ void combo_b_kernel(T *__restrict__ x, MArgs<T> a, const double2 *__restrict__ g, int64_t n) {
    using R = typename RealB<T>::type;
    const int r = blockIdx.y;
    const size_t off = (size_t)r * n;
    __shared__ R cr[32], ci[32];
    if (threadIdx.x < a.k) {
        cr[threadIdx.x] = (R)g[r * a.k + threadIdx.x].x;
        ci[threadIdx.x] = (R)g[r * a.k + threadIdx.x].y;
    }
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n / Pack<T>::N; i += (int64_t)gridDim.x * blockDim.x) {
        Pack<T> v = ldp<T>(x + off, i);
#pragma unroll 8
        for (int j = 0; j < a.k; ++j) {
            const Pack<T> u = ldp(a.v[j] + off, i);
#pragma unroll
            for (int e = 0; e < Pack<T>::N; ++e) {
                cadd_prod(v.e[e], mk<R>(cr[j], ci[j]), u.e[e]);
            }
        }
        stp(x + off, i, v);
    }
}

// x_r += sum_j g_j Z_j,r for the k (<= 32) stored normal-equations residuals
// z_0 .. z_{k-1} of k CGNR iterations, with g the solution's coefficients in
// that basis: x = sum_k a_k p_k and p_k = z_k + b_{k-1} p_{k-1} give
// g_{k-1} = a_{k-1}, g_j = a_j + b_j g_{j+1}, where a_j = |z_j|^2 / |w_j|^2
// and b_j = |z_{j+1}|^2 / |z_j|^2 come from the scalar slots zb + j and wb + j.
// directions: the Z_j are the p_j themselves, g_j = a_j.
template <typename T>
__global__ void cg_combine_b_kernel(T *__restrict__ x, MArgs<T> a, const double *__restrict__ s, int base, int stride,
                                    int zb, int wb, int directions, int64_t n) {
    using R = typename RealB<T>::type;
    __shared__ R gam[32];
    __shared__ double al[32], be[32];
    const int r = blockIdx.y;
    const size_t off = (size_t)r * n;
    if (threadIdx.x < a.k) {  // the divisions side by side, the recurrence by one thread
        const int j = threadIdx.x;
        const double *sr = s + base + (size_t)r * stride;
        const double zz = sr[zb + j], ww = sr[wb + j];
        al[j] = ww > 0.0 ? zz / ww : 0.0;
        be[j] = (!directions && j + 1 < a.k && zz > 0.0) ? sr[zb + j + 1] / zz : 0.0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double g = 0.0;
        for (int j = a.k - 1; j >= 0; --j) {
            g = al[j] + be[j] * g;
            gam[j] = (R)g;
        }
    }
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n / Pack<T>::N; i += (int64_t)gridDim.x * blockDim.x) {
        Pack<T> v = ldp<T>(x + off, i);
#pragma unroll 8
        for (int j = 0; j < a.k; ++j) {
            const Pack<T> u = ldp(a.v[j] + off, i);
#pragma unroll
            for (int e = 0; e < Pack<T>::N; ++e) {
                v.e[e].x += gam[j] * u.e[e].x;
                v.e[e].y += gam[j] * u.e[e].y;
            }
        }
        stp(x + off, i, v);
    }
}

// End of a chunk of m CGNR iterations k0 .. k0+m-1 that kept the residuals
// z_{k0+1} .. z_{k0+m-1} (and z_{k0+m} when the chunk is not the last) and
// carried w = D p by recursion.  With p_0 the chunk's first direction,
// p_t = z_t + b_{t-1} p_{t-1}:
//   x (+)= sum_t a_t p_t = G_0 p_0 + sum_{t=1}^{m-1} G_t z_t,
//          G_{m-1} = a_{m-1}, G_t = a_t + b_t G_{t+1};
//   p_0 <- p_m = P_0 p_0 + sum_{t=1}^{m} P_t z_t, P_m = 1, P_t = b_t P_{t+1}
// (the latter only with next).  a_t = |z_t|^2 / |w_t|^2 and
// b_t = |z_{t+1}|^2 / |z_t|^2 from the ring of scalar slots
// zb + (k0 + t) % rs and wb + (k0 + t) % rs.
template <typename T>
__global__ void cg_chunk_b_kernel(T *__restrict__ x, T *__restrict__ p, MArgs<T> z, const double *__restrict__ s,
                                  int base, int stride, int zb, int wb, int k0, int rs, int m, int next, int xinit,
                                  int64_t n) {
    using R = typename RealB<T>::type;
    __shared__ R G[33], P[33];
    __shared__ double al[32], be[32];
    const int r = blockIdx.y;
    const size_t off = (size_t)r * n;
    if (threadIdx.x < m) {  // the divisions side by side, the recurrences by one thread
        const int t = threadIdx.x;
        const double *sr = s + base + (size_t)r * stride;
        const double zt = sr[zb + (k0 + t) % rs], wt = sr[wb + (k0 + t) % rs];
        al[t] = wt > 0.0 ? zt / wt : 0.0;
        be[t] = ((t + 1 < m || next) && zt > 0.0) ? sr[zb + (k0 + t + 1) % rs] / zt : 0.0;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double g = 0.0, q = 1.0;
        if (next) P[m] = (R)1;
        for (int t = m - 1; t >= 0; --t) {
            g = al[t] + (t + 1 < m ? be[t] * g : 0.0);
            G[t] = (R)g;
            if (next) {
                q *= be[t];
                P[t] = (R)q;
            }
        }
    }
    __syncthreads();
    const R p0 = next ? P[0] : R(0);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n / Pack<T>::N; i += (int64_t)gridDim.x * blockDim.x) {
        const Pack<T> pv = ldp<T>(p + off, i);
        Pack<T> xv, pn;
        if (xinit) {
#pragma unroll
            for (int e = 0; e < Pack<T>::N; ++e) xv.e[e] = T{0, 0};
        } else {
            xv = ldp<T>(x + off, i);
        }
#pragma unroll
        for (int e = 0; e < Pack<T>::N; ++e) {
            pn.e[e].x = p0 * pv.e[e].x;
            pn.e[e].y = p0 * pv.e[e].y;
            xv.e[e].x += G[0] * pv.e[e].x;
            xv.e[e].y += G[0] * pv.e[e].y;
        }
#pragma unroll 8
        for (int t = 1; t < m; ++t) {
            const Pack<T> u = ldp(z.v[t - 1] + off, i);
#pragma unroll
            for (int e = 0; e < Pack<T>::N; ++e) {
                xv.e[e].x += G[t] * u.e[e].x;
                xv.e[e].y += G[t] * u.e[e].y;
                pn.e[e].x += P[t] * u.e[e].x;  // (not used by the last chunk)
                pn.e[e].y += P[t] * u.e[e].y;
            }
        }
        stp(x + off, i, xv);
        if (next) {
            const Pack<T> u = ldp(z.v[m - 1] + off, i);
#pragma unroll
            for (int e = 0; e < Pack<T>::N; ++e) {
                pn.e[e].x += u.e[e].x;  // P_m = 1
                pn.e[e].y += u.e[e].y;
            }
            stp(p + off, i, pn);
        }
    }
}

// p = zt + c (p - z), c = s[izt] / s[iz] (0 where the denominator is not positive)
template <typename T>
__global__ void cg_redirect_kernel(T *__restrict__ p, const T *__restrict__ zt, const T *__restrict__ z,
                                   const double *__restrict__ s, int izt, int iz, int64_t n) {
    using R = typename RealB<T>::type;
    const R cf = s[iz] > 0.0 ? (R)(s[izt] / s[iz]) : R(0);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const T pv = p[i], zv = z[i], tv = zt[i];
        T o;
        o.x = tv.x + cf * (pv.x - zv.x);
        o.y = tv.y + cf * (pv.y - zv.y);
        p[i] = o;
    }
}

// CTAs per right-hand side: one pass of 16 bytes per thread up to cap_per_sm
// CTAs per SM over all right-hand sides
template <typename T> dim3 grid_b(dwf_ctx *c, int64_t n, int nrhs, int cap_per_sm) {
    int64_t b = (n + BT * Pack<T>::N - 1) / (BT * Pack<T>::N);
    int64_t cap = std::max<int64_t>(1, (int64_t)c->sm_count * cap_per_sm / std::max(1, nrhs));
    cap = std::min<int64_t>(cap, 1024);  // partial-sum buffers hold 1024 blocks per value
    return dim3((unsigned)std::max<int64_t>(1, std::min(b, cap)), (unsigned)nrhs);
}

// ... and of a reduction: fewer CTAs, at least four passes each, since every one
// of them ends with a ticket on one address
template <typename T> dim3 grid_r(dwf_ctx *c, int64_t n, int nrhs) {
    dim3 g = grid_b<T>(c, n, nrhs, 8);
    const int64_t b = (n + BT * Pack<T>::N * 4 - 1) / (BT * Pack<T>::N * 4);
    g.x = (unsigned)std::max<int64_t>(1, std::min<int64_t>(g.x, std::max<int64_t>(b, c->sm_count / nrhs)));
    return g;
}

}  // namespace

// Buffers of batched reductions: partial sums [nrhs][8][blocks] and counters.
void BatchScratch::ensure(int nrhs) {
    size_t need = sizeof(double2) * (size_t)nrhs * 8 * 1024;
    if (part.bytes < need) part.alloc(need);
    if (count.bytes < sizeof(unsigned) * (size_t)nrhs) {
        count.alloc(sizeof(unsigned) * (size_t)nrhs);
        DWF_CUDA(cudaMemset(count.p, 0, count.bytes));
    }
}

template <typename T> void norm2_b(dwf_ctx *c, BatchScratch &bs, int base, int stride, const T *x, int64_t n, int nrhs) {
    dim3 g = grid_r<T>(c, n, nrhs);
    norm2_b_kernel<T><<<g, BT, 0, c->stream>>>(x, n, bs.part.as<double>(), bs.count.as<unsigned>(), c->scal.as<double>(),
                                               base, stride);
    DWF_CHECK_LAUNCH();
}

template <typename T>
void multidot_b(dwf_ctx *c, BatchScratch &bs, int base, int stride, T *const *V, int k, const T *w, int64_t n, int nrhs) {
    dim3 g = grid_r<T>(c, n, nrhs);
    for (int j0 = 0; j0 < k; j0 += 8) {
        int kk = std::min(8, k - j0);
#define MDB(K)                                                                                              \
    {                                                                                                       \
        VArgs<T, K> a;                                                                                      \
        for (int j = 0; j < K; ++j) a.v[j] = V[j0 + j];                                                     \
        multidot_b_kernel<T, K><<<g, BT, 0, c->stream>>>(a, w, n, bs.part.as<double>(), bs.count.as<unsigned>(), \
                                                         c->scal.as<double>(), base + 2 * j0, stride);      \
    }
        switch (kk) {
            case 1: MDB(1) break;
            case 2: MDB(2) break;
            case 3: MDB(3) break;
            case 4: MDB(4) break;
            case 5: MDB(5) break;
            case 6: MDB(6) break;
            case 7: MDB(7) break;
            default: MDB(8) break;
        }
#undef MDB
        DWF_CHECK_LAUNCH();
    }
}

template <typename T>
void multiaxpy_b(dwf_ctx *c, T *w, T *const *V, int k, int base, int stride, double sgn, int64_t n, int nrhs) {
    dim3 g = grid_b<T>(c, n, nrhs, 16);
    for (int j0 = 0; j0 < k; j0 += 32) {
        MArgs<T> a;
        a.k = std::min(32, k - j0);
        for (int j = 0; j < a.k; ++j) a.v[j] = V[j0 + j];
        multiaxpy_b_kernel<T><<<g, BT, 0, c->stream>>>(w, a, c->scal.as<double>(), base + 2 * j0, stride, sgn, n);
        DWF_CHECK_LAUNCH();
    }
}

template <typename T>
void cg_r_b(dwf_ctx *c, T *r, const T *rin, const T *w, int base, int stride, int izz, int iww, int64_t n, int nrhs) {
    dim3 g = grid_b<T>(c, n, nrhs, 16);
    launch_after(cg_r_b_kernel<T>, g, dim3(BT), 0, c->stream, r, rin, w, c->scal.as<double>(), base, stride, izz, iww, n);
    DWF_CHECK_LAUNCH();
}

template <typename T>
void cg_p_b(dwf_ctx *c, T *pout, const T *pin, const T *z, int base, int stride, int izz, int inew, int64_t n, int nrhs) {
    dim3 g = grid_b<T>(c, n, nrhs, 16);
    launch_after(cg_p_b_kernel<T>, g, dim3(BT), 0, c->stream, pout, pin, z, c->scal.as<double>(), base, stride, izz, inew, n);
    DWF_CHECK_LAUNCH();
}

template <typename T>
void cg_px_b(dwf_ctx *c, T *x, T *pout, const T *pin, const T *z, int base, int stride, int izz, int iww, int inew,
             int64_t n, int nrhs, bool last, bool xinit) {
    dim3 g = grid_b<T>(c, n, nrhs, 16);
    cg_px_b_kernel<T><<<g, BT, 0, c->stream>>>(x, pout, pin, z, c->scal.as<double>(), base, stride, izz, iww, inew,
                                               n, last ? 1 : 0, xinit ? 1 : 0);
    DWF_CHECK_LAUNCH();
}

template <typename T>
void cg_pxd_b(dwf_ctx *c, T *x, T *pout, const T *pin, T *const *pend, int np, const T *z, int base, int stride,
              int izz, int iww, int inew, int ia, int64_t n, int nrhs, int mode) {
    DWF_REQUIRE(mode >= 0 && mode <= 2 && np >= 0 && np <= CG_MAXDEFER && !(mode == 0 && np == CG_MAXDEFER),
                DWF_EINVAL, "cg_pxd_b: mode or pending count");
    dim3 g = grid_b<T>(c, n, nrhs, 16);
    Pending<T> pd{};
    for (int j = 0; j < np; ++j) pd.p[j] = pend[j];
    double *s = c->scal.as<double>();
#define PX(NP) cg_pxd_b_kernel<T, NP><<<g, BT, 0, c->stream>>>(x, pout, pin, pd, z, s, base, stride, izz, iww, inew, ia, \
                                                                n, mode)
    switch (np) {
        case 0: PX(0); break;
        case 1: PX(1); break;
        case 2: PX(2); break;
        default: PX(3); break;
    }
#undef PX
    DWF_CHECK_LAUNCH();
}

template <typename T>
void normalised_b(dwf_ctx *c, double2 *out, const T *x, int base, int stride, int64_t n, int nrhs) {
    dim3 g = grid_b<T>(c, n, nrhs, 16);
    normalised_b_kernel<T><<<g, BT, 0, c->stream>>>(out, x, c->scal.as<double>(), base, stride, n);
    DWF_CHECK_LAUNCH();
}

template <typename T> void gcr_wr_b(dwf_ctx *c, T *w, T *res, const GcrStep &step, int64_t n, int nrhs) {
    DWF_REQUIRE(nrhs <= 32, DWF_EINVAL, "GCR step: at most 32 right-hand sides");
    dim3 g = grid_b<T>(c, n, nrhs, 16);
    gcr_wr_b_kernel<T><<<g, BT, 0, c->stream>>>(w, res, step, n);
    DWF_CHECK_LAUNCH();
}

template <typename T> void combo_b(dwf_ctx *c, T *x, T *const *V, int k, const double2 *g, int64_t n, int nrhs) {
    DWF_REQUIRE(k <= 32, DWF_EINVAL, "combo_b: at most 32 vectors");
    if (k == 0) return;
    dim3 gr = grid_b<T>(c, n, nrhs, 16);
    MArgs<T> a;
    a.k = k;
    for (int j = 0; j < k; ++j) a.v[j] = V[j];
    combo_b_kernel<T><<<gr, BT, 0, c->stream>>>(x, a, g, n);
    DWF_CHECK_LAUNCH();
}

template <typename T>
void cg_combine_b(dwf_ctx *c, T *x, T *const *Z, int k, int base, int stride, int zb, int wb, bool directions, int64_t n,
                  int nrhs) {
    DWF_REQUIRE(k >= 1 && k <= 32, DWF_EINVAL, "cg_combine_b: 1 to 32 stored fields");
    dim3 gr = grid_b<T>(c, n, nrhs, 16);
    MArgs<T> a;
    a.k = k;
    for (int j = 0; j < k; ++j) a.v[j] = Z[j];
    cg_combine_b_kernel<T><<<gr, BT, 0, c->stream>>>(x, a, c->scal.as<double>(), base, stride, zb, wb, directions ? 1 : 0, n);
    DWF_CHECK_LAUNCH();
}

template <typename T>
void cg_chunk_b(dwf_ctx *c, T *x, T *p, T *const *Z, int m, bool next, bool xinit, int base, int stride, int zb, int wb,
                int k0, int rs, int64_t n, int nrhs) {
    DWF_REQUIRE(m >= 1 && m <= 32 && rs > m, DWF_EINVAL, "cg_chunk_b: 1 to 32 iterations, slot ring longer than that");
    dim3 gr = grid_b<T>(c, n, nrhs, 16);
    MArgs<T> a;
    a.k = next ? m : m - 1;
    for (int j = 0; j < a.k; ++j) a.v[j] = Z[j];
    cg_chunk_b_kernel<T><<<gr, BT, 0, c->stream>>>(x, p, a, c->scal.as<double>(), base, stride, zb, wb, k0, rs, m,
                                                   next ? 1 : 0, xinit ? 1 : 0, n);
    DWF_CHECK_LAUNCH();
}

template <typename T>
void cg_redirect(dwf_ctx *c, T *p, const T *zt, const T *z, int izt, int iz, int64_t n) {
    cg_redirect_kernel<T><<<grid_b<T>(c, n, 1, 16), BT, 0, c->stream>>>(p, zt, z, c->scal.as<double>(), izt, iz, n);
    DWF_CHECK_LAUNCH();
}

#define INSTB(T)                                                                                            \
    template void norm2_b<T>(dwf_ctx *, BatchScratch &, int, int, const T *, int64_t, int);                  \
    template void multidot_b<T>(dwf_ctx *, BatchScratch &, int, int, T *const *, int, const T *, int64_t, int); \
    template void multiaxpy_b<T>(dwf_ctx *, T *, T *const *, int, int, int, double, int64_t, int);            \
    template void cg_r_b<T>(dwf_ctx *, T *, const T *, const T *, int, int, int, int, int64_t, int);          \
    template void cg_p_b<T>(dwf_ctx *, T *, const T *, const T *, int, int, int, int, int64_t, int);          \
    template void cg_px_b<T>(dwf_ctx *, T *, T *, const T *, const T *, int, int, int, int, int, int64_t, int, bool, \
                             bool);                                                                            \
    template void cg_pxd_b<T>(dwf_ctx *, T *, T *, const T *, T *const *, int, const T *, int, int, int, int, int, \
                              int, int64_t, int, int);                                                         \
    template void cg_combine_b<T>(dwf_ctx *, T *, T *const *, int, int, int, int, int, bool, int64_t, int);  \
    template void cg_chunk_b<T>(dwf_ctx *, T *, T *, T *const *, int, bool, bool, int, int, int, int, int, int,   \
                                int64_t, int);                                                                 \
    template void normalised_b<T>(dwf_ctx *, double2 *, const T *, int, int, int64_t, int);                   \
    template void cg_redirect<T>(dwf_ctx *, T *, const T *, const T *, int, int, int64_t);                   \
    template void gcr_wr_b<T>(dwf_ctx *, T *, T *, const GcrStep &, int64_t, int);                           \
    template void combo_b<T>(dwf_ctx *, T *, T *const *, int, const double2 *, int64_t, int);
INSTB(float2)
INSTB(double2)

}  // namespace dwf
