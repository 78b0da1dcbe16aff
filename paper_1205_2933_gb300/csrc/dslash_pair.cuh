// FP32 fine Dslash with two fifth-dimension slices per thread, written for any
// even Ls up to 64 and instantiated for 4, 6, 8, 10, 12, 16, 20, 24, 32, 48 and
// 64 (each includer has some of them).  Every other Ls takes the one-slice kernel
// of dslash.cu, slower and without these epilogues.
//
// Same operator as dslash.cu (Sec. 2: Shamir domain-wall operator; Sec. 4:
// 11-site stencil).  A thread owns the slices s0 = 2j and s1 = 2j + 1 of one
// 4D site.  Every complex quantity is held as two register pairs: the real
// parts (s0, s1) and the imaginary parts (s0, s1).  The link is the same
// for both slices, so each complex multiply-add of the 3x3 link products is
// four packed FP32x2 FMAs for the two slices (fma.rn.f32x2) instead of eight
// scalar FMAs, and multiplications by +-i are a choice of operands, not
// arithmetic.  Component loads are 16 bytes (the two slices of one
// component are adjacent in the s-fastest layout).  Links are staged once
// per CTA in shared memory, scaled by their hop coefficient; one 16-byte load
// brings two of a link's elements, which are duplicated into packed
// operands.  The fifth-dimension neighbours come from the thread's own pair
// and from the neighbouring lane (warp shuffles).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "dslash_norm.cuh"

namespace dwf {

namespace {

struct P2 {
    unsigned long long v;
};

__device__ __forceinline__ P2 pk(float a, float b) {
    P2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpk(P2 p) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(p.v));
    return r;
}
__device__ __forceinline__ P2 fma2(P2 a, P2 b, P2 c) {
    P2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ P2 add2(P2 a, P2 b) {
    P2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ P2 sub2(P2 a, P2 b) {
    P2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ P2 mul2(P2 a, P2 b) {
    P2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

// a complex number for the two slices: real parts and imaginary parts
struct CP {
    P2 re, im;
};

// the half-spinor rows of (1 + sig g_mu) p for both slices; p[k] holds
// component k = spin*3 + colour as (re_s0, im_s0, re_s1, im_s1)
template <int MU>
__device__ __forceinline__ void project2(const float4 p[12], float sig, CP h[6]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float4 p0 = p[a], p1 = p[3 + a], p2 = p[6 + a], p3 = p[9 + a];
        if (MU == 0) {  // h0 = p0 + sig i p3, h1 = p1 + sig i p2
            h[a].re = pk(p0.x - sig * p3.y, p0.z - sig * p3.w);
            h[a].im = pk(p0.y + sig * p3.x, p0.w + sig * p3.z);
            h[3 + a].re = pk(p1.x - sig * p2.y, p1.z - sig * p2.w);
            h[3 + a].im = pk(p1.y + sig * p2.x, p1.w + sig * p2.z);
        } else if (MU == 1) {  // h0 = p0 - sig p3, h1 = p1 + sig p2
            h[a].re = pk(p0.x - sig * p3.x, p0.z - sig * p3.z);
            h[a].im = pk(p0.y - sig * p3.y, p0.w - sig * p3.w);
            h[3 + a].re = pk(p1.x + sig * p2.x, p1.z + sig * p2.z);
            h[3 + a].im = pk(p1.y + sig * p2.y, p1.w + sig * p2.w);
        } else if (MU == 2) {  // h0 = p0 + sig i p2, h1 = p1 - sig i p3
            h[a].re = pk(p0.x - sig * p2.y, p0.z - sig * p2.w);
            h[a].im = pk(p0.y + sig * p2.x, p0.w + sig * p2.z);
            h[3 + a].re = pk(p1.x + sig * p3.y, p1.z + sig * p3.w);
            h[3 + a].im = pk(p1.y - sig * p3.x, p1.w - sig * p3.z);
        } else {  // h0 = p0 + sig p2, h1 = p1 + sig p3
            h[a].re = pk(p0.x + sig * p2.x, p0.z + sig * p2.z);
            h[a].im = pk(p0.y + sig * p2.y, p0.w + sig * p2.w);
            h[3 + a].re = pk(p1.x + sig * p3.x, p1.z + sig * p3.z);
            h[3 + a].im = pk(p1.y + sig * p3.y, p1.w + sig * p3.w);
        }
    }
}

// acc += (1 + sig g_mu) rebuilt from the link products u (rows 0, 1):
//   g_x: row2 = -sig i u1, row3 = -sig i u0     g_y: row2 = sig u1, row3 = -sig u0
//   g_z: row2 = -sig i u0, row3 =  sig i u1     g_t: row2 = sig u0, row3 =  sig u1
// with -i u = (u.im, -u.re) and i u = (-u.im, u.re).
template <int MU>
__device__ __forceinline__ void recon2(CP acc[12], int a, const CP &u0, const CP &u1, float sig) {
    acc[a].re = add2(acc[a].re, u0.re);
    acc[a].im = add2(acc[a].im, u0.im);
    acc[3 + a].re = add2(acc[3 + a].re, u1.re);
    acc[3 + a].im = add2(acc[3 + a].im, u1.im);
    const bool pos = sig > 0.f;
    CP &r2 = acc[6 + a], &r3 = acc[9 + a];
    if (MU == 0) {  // row2 += -sig i u1 = sig (u1.im, -u1.re); row3 += sig (u0.im, -u0.re)
        if (pos) { r2.re = add2(r2.re, u1.im); r2.im = sub2(r2.im, u1.re); r3.re = add2(r3.re, u0.im); r3.im = sub2(r3.im, u0.re); }
        else     { r2.re = sub2(r2.re, u1.im); r2.im = add2(r2.im, u1.re); r3.re = sub2(r3.re, u0.im); r3.im = add2(r3.im, u0.re); }
    } else if (MU == 1) {  // row2 += sig u1; row3 -= sig u0
        if (pos) { r2.re = add2(r2.re, u1.re); r2.im = add2(r2.im, u1.im); r3.re = sub2(r3.re, u0.re); r3.im = sub2(r3.im, u0.im); }
        else     { r2.re = sub2(r2.re, u1.re); r2.im = sub2(r2.im, u1.im); r3.re = add2(r3.re, u0.re); r3.im = add2(r3.im, u0.im); }
    } else if (MU == 2) {  // row2 += sig (u0.im, -u0.re); row3 += sig (-u1.im, u1.re)
        if (pos) { r2.re = add2(r2.re, u0.im); r2.im = sub2(r2.im, u0.re); r3.re = sub2(r3.re, u1.im); r3.im = add2(r3.im, u1.re); }
        else     { r2.re = sub2(r2.re, u0.im); r2.im = add2(r2.im, u0.re); r3.re = add2(r3.re, u1.im); r3.im = sub2(r3.im, u1.re); }
    } else {  // row2 += sig u0; row3 += sig u1
        if (pos) { r2.re = add2(r2.re, u0.re); r2.im = add2(r2.im, u0.im); r3.re = add2(r3.re, u1.re); r3.im = add2(r3.im, u1.im); }
        else     { r2.re = sub2(r2.re, u0.re); r2.im = sub2(r2.im, u0.im); r3.re = sub2(r3.re, u1.re); r3.im = sub2(r3.im, u1.im); }
    }
}

// One 4D hop for both slices from the neighbour's preloaded row p (the 12
// components of the thread's two slices).  sL: the staged link (9 elements
// (re, im), hop coefficient included; each part is duplicated in registers);
// ADJ: use its adjoint.
template <int MU, bool ADJ>
__device__ __forceinline__ void hop2(CP acc[12], const float4 p[12], const float2 *sL, float sig) {
    float2 lk[10];
#pragma unroll
    for (int e = 0; e < 5; ++e) { const float4 q = *reinterpret_cast<const float4 *>(sL + 2 * e); lk[2 * e] = make_float2(q.x, q.y); lk[2 * e + 1] = make_float2(q.z, q.w); }
    CP h[6];
    project2<MU>(p, sig, h);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        // u[sp] = sum_b M(a,b) h[sp][b]; M = U (a,b) or conj(U (b,a))
        P2 rp0 = pk(0.f, 0.f), rn0 = rp0, ip0 = rp0, in0 = rp0;
        P2 rp1 = rp0, rn1 = rp0, ip1 = rp0, in1 = rp0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const float2 m = ADJ ? lk[b * 3 + a] : lk[a * 3 + b];
            const P2 mre = pk(m.x, m.x), mim = pk(m.y, m.y);
            const CP &h0 = h[b], &h1 = h[3 + b];
            if (!ADJ) {  // (mre + i mim)(h.re + i h.im)
                rp0 = fma2(mre, h0.re, rp0); rn0 = fma2(mim, h0.im, rn0);
                ip0 = fma2(mre, h0.im, ip0); ip0 = fma2(mim, h0.re, ip0);
                rp1 = fma2(mre, h1.re, rp1); rn1 = fma2(mim, h1.im, rn1);
                ip1 = fma2(mre, h1.im, ip1); ip1 = fma2(mim, h1.re, ip1);
            } else {     // (mre - i mim)(h.re + i h.im)
                rp0 = fma2(mre, h0.re, rp0); rp0 = fma2(mim, h0.im, rp0);
                ip0 = fma2(mre, h0.im, ip0); in0 = fma2(mim, h0.re, in0);
                rp1 = fma2(mre, h1.re, rp1); rp1 = fma2(mim, h1.im, rp1);
                ip1 = fma2(mre, h1.im, ip1); in1 = fma2(mim, h1.re, in1);
            }
        }
        CP u0, u1;
        if (!ADJ) {
            u0.re = sub2(rp0, rn0); u0.im = ip0;
            u1.re = sub2(rp1, rn1); u1.im = ip1;
        } else {
            u0.re = rp0; u0.im = sub2(ip0, in0);
            u1.re = rp1; u1.im = sub2(ip1, in1);
        }
        recon2<MU>(acc, a, u0, u1, sig);
    }
}

// the 12 components of a thread's two slices in one site's row
template <int LS> __device__ __forceinline__ void ldrow(float4 p[12], const float2 *row) {
#pragma unroll
    for (int k = 0; k < 12; ++k) p[k] = *reinterpret_cast<const float4 *>(row + k * LS);
}

// L2 priority of data that nobody reads again soon (first) or of any other
__device__ __forceinline__ uint64_t l2_policy(int first) {
    uint64_t f, n;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(f));
    asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(n));
    return first ? f : n;
}

__device__ __forceinline__ float4 ld_hint(const float4 *p, uint64_t policy) {
    float4 v;
    asm volatile("ld.global.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p), "l"(policy));
    return v;
}

__device__ __forceinline__ void st_hint(float4 *p, const float4 &v, uint64_t policy) {
    asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z),
                 "f"(v.w), "l"(policy) : "memory");
}

// A warp holds 32 / (LS/2) whole sites (LS/2 lanes each, the lanes left over
// idle), so that the fifth-dimension neighbours are lanes of the same warp.
// A staged link takes 10 float2 (9 used) and a site LSTRIDE: the sites of one
// warp start 4 banks apart and their reads of the same elements do not collide.
//
// What bounds the kernel is the L1 data path, 76 % of its wavefronts busy when
// four fields of 16^3 x 32 x 16 took 450 us, 69 % at the 412 us they take now
// (DRAM at 242 / 412 = 59 % of the copy rate): nine
// rows of 96 bytes per 5D site are read, and the rows in flight (16 warps x 2)
// exceed L1, so 87 % of them are also filled whatever the shape of the CTA's
// sites.  Hence: the links as 16-byte loads of two elements instead of one
// element with both parts duplicated (443 -> 419 us), two right-hand sides per
// staged link (from Ls 10 on four leave too few CTAs in small grids, 12 % slower
// at 5040 sites x 3 x Ls 12; dslash_pair_ls has the rule), and the second field of the fused kernels asked for by an L2 prefetch
// and loaded while the last hop computes, which leaves shared memory to L1 and
// lets them share links as well (362 -> 333 us for 12 fields of 12^3 x 16 x 16
// against staging it by cp.async).  The CTA's sites are a brick (Brick) so that
// no extent wastes lanes; bricks of equal size measured within 2 %.
constexpr int LSTRIDE = 82;

// 4D coordinates of site ls of the brick `bid`; false outside of the brick or the lattice
__device__ __forceinline__ bool brick_site(const Brick &k, const Geom &g, unsigned bid, unsigned ls, int x[4]) {
    unsigned q = k.dn[0].div(bid);
    x[0] = (bid - q * k.dn[0].d) * k.b[0];
    bid = q;
    q = k.dn[1].div(bid);
    x[1] = (bid - q * k.dn[1].d) * k.b[1];
    bid = q;
    q = k.dn[2].div(bid);
    x[2] = (bid - q * k.dn[2].d) * k.b[2];
    x[3] = q * k.b[3];
    q = k.db[0].div(ls);
    x[0] += ls - q * k.b[0];
    ls = q;
    q = k.db[1].div(ls);
    x[1] += ls - q * k.b[1];
    ls = q;
    q = k.db[2].div(ls);
    x[2] += ls - q * k.b[2];
    x[3] += q;
    return (int)q < k.b[3] && x[0] < g.L[0] && x[1] < g.L[1] && x[2] < g.L[2] && x[3] < g.L[3];
}

__device__ __forceinline__ int site_of(const Geom &g, const int x[4]) {
    return ((x[3] * g.L[2] + x[2]) * g.L[1] + x[1]) * g.L[0] + x[0];
}

constexpr int PAIR_THREADS = 128;  // at most; 128 registers per thread

// A CTA stages its sites' links once and applies the operator to rb
// right-hand sides in turn (r = blockIdx.y * rb + 0 .. rb-1, below nrhs).
// EPI 0: out = D in (or D^+ in).  EPI 1: also |out_r|^2 of every right-hand
// side r: one FP64 partial per CTA (FP32 per warp), see dslash_norm.cuh.
// EPI 2: out = zu.zin - a D^+ in, and |out_r|^2 as with EPI 1.
// EPI 3: out = zu.zin - D in (a residual b - D x), no norm.
// EPI 4: out = D in + a zu.zin (CGNR's w = D p carried as D z + b w), and |out_r|^2.
// a = zz[r * stride] / ww[r * stride] (0 where the denominator is not positive).
template <bool DAG, int LS, int EPI>
__global__ void __launch_bounds__(PAIR_THREADS, 4)
dslash_pair_kernel(float2 *out0, const float2 *in0, const float2 *__restrict__ U, Geom g,
                   Brick bk, float diag, float mf, int64_t field, NormOut nout, ZUpdate zu, int nrhs, int rb) {
    constexpr bool NORM = EPI == 1 || EPI == 2 || EPI == 4;
    constexpr int TPS = LS / 2;      // lanes per site
    constexpr int SPW = 32 / TPS;    // sites per warp
    constexpr int row = 12 * LS;
    extern __shared__ __align__(16) float2 sL[];  // [sites][LSTRIDE]
    const int spb = (blockDim.x >> 5) * SPW;
    const int r0 = blockIdx.y * rb, r1 = min(r0 + rb, nrhs);
    const int lane = threadIdx.x & 31, wl = lane / TPS, j = lane - wl * TPS;
    const int ls = (threadIdx.x >> 5) * SPW + wl, s0 = 2 * j;
    int x[4];
    const bool active = brick_site(bk, g, blockIdx.x, ls, x) && wl < SPW;
    if (!active) x[0] = x[1] = x[2] = x[3] = 0;  // idle lanes compute on site 0 and store nothing
    const int site = site_of(g, x);
    // the links of the CTA's sites: U_mu(x) and U_mu(x-mu), two stored rows, the
    // third rebuilt as conj(row0 x row1) (det U = 1), scaled by the hop
    // coefficient, (re, im) per element
    for (int jj = threadIdx.x; jj < spb * 8; jj += blockDim.x) {
        const int k = jj & 7, mu = k & 3;
        int y[4];
        if (brick_site(bk, g, blockIdx.x, jj >> 3, y)) {
            bool wrap = k < 4 ? y[mu] == g.L[mu] - 1 : y[mu] == 0;
            if (k >= 4) y[mu] = wrap ? g.L[mu] - 1 : y[mu] - 1;
            const float2 *p = U + ((size_t)site_of(g, y) * 4 + mu) * 6;
            float2 m[9];
#pragma unroll
            for (int e = 0; e < 6; ++e) m[e] = p[e];
            m[6] = conj2(cmul(m[1], m[5]) - cmul(m[2], m[4]));
            m[7] = conj2(cmul(m[2], m[3]) - cmul(m[0], m[5]));
            m[8] = conj2(cmul(m[0], m[4]) - cmul(m[1], m[3]));
            const float coef = (mu == 3 && g.ap && wrap) ? 0.5f : -0.5f;
#pragma unroll
            for (int e = 0; e < 9; ++e) {
                const float re = coef * m[e].x, im = coef * m[e].y;
                sL[(jj >> 3) * LSTRIDE + k * 10 + e] = make_float2(re, im);
            }
        }
    }
    // the neighbour's row, fw: x + mu, else x - mu
    const int strd[4] = {1, g.L[0], g.L[0] * g.L[1], g.L[0] * g.L[1] * g.L[2]};
    const size_t self_off = (size_t)site * row + s0;
    auto nb = [&](int mu, bool fw) {
        const int step = fw ? (x[mu] == g.L[mu] - 1 ? -x[mu] : 1) : (x[mu] == 0 ? g.L[mu] - 1 : -1);
        return (size_t)(site + step * strd[mu]) * row + s0;
    };
    // EPI >= 2: the second field's components are asked for ahead, into L2, and
    // loaded while the last hop computes
    auto request_z = [&](int r) {
        const float2 *zp = zu.zin + (size_t)r * (size_t)field + self_off;
#pragma unroll
        for (int k = 0; k < 12; ++k) asm volatile("prefetch.global.L2 [%0];\n" ::"l"(zp + k * LS));
    };
    pdl_wait();  // the links are constant; fields and scalar slots are not
    if (EPI >= 2 && active) request_z(r0);
    __syncthreads();
    for (int rhs = r0; rhs < r1; ++rhs) {
        const float2 *in = in0 + (size_t)rhs * (size_t)field;
        float2 *out = out0 + (size_t)rhs * (size_t)field;
        // the first two hops' rows are requested together with the thread's own
        // row; each later row is requested while the hop before it computes
        float4 pa[12], pb[12], self[12];
        ldrow<LS>(pa, in + nb(0, true));
        ldrow<LS>(pb, in + nb(0, false));
        ldrow<LS>(self, in + self_off);
        // fifth dimension.  D: -P_- psi(s+1) (components 6..11), -P_+ psi(s-1)
        // (components 0..5), wrapping with +mf.  D^+: the two projectors swap.
        const int up_lo = DAG ? 0 : 6, dn_lo = DAG ? 6 : 0;
        const int base = lane - j;
        const int lnext = base + (j == TPS - 1 ? 0 : j + 1);
        const int lprev = base + (j == 0 ? TPS - 1 : j - 1);
        const float c_up1 = (s0 + 1 == LS - 1) ? mf : -1.f;  // s1 + 1 wraps to s = 0
        const float c_dn0 = (s0 == 0) ? mf : -1.f;           // s0 - 1 wraps to s = Ls-1
        // (diag psi joins them in one fused operation: rounded on its own, the largest
        // term of the sum would raise the kernel's error by 4 %)
        CP acc[12];
        const P2 dg = pk(diag, diag);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            // from s+1: slice s0 takes own s1 (coefficient -1), slice s1 takes s0 of the next lane
            const float4 su = self[up_lo + q];
            const float nx = __shfl_sync(0xffffffffu, su.x, lnext), ny = __shfl_sync(0xffffffffu, su.y, lnext);
            acc[up_lo + q].re = fma2(dg, pk(su.x, su.z), pk(-su.z, c_up1 * nx));
            acc[up_lo + q].im = fma2(dg, pk(su.y, su.w), pk(-su.w, c_up1 * ny));
            // from s-1: slice s0 takes s1 of the previous lane, slice s1 takes own s0 (coefficient -1)
            const float4 sd = self[dn_lo + q];
            const float pz = __shfl_sync(0xffffffffu, sd.z, lprev), pw = __shfl_sync(0xffffffffu, sd.w, lprev);
            acc[dn_lo + q].re = fma2(dg, pk(sd.x, sd.z), pk(c_dn0 * pz, -sd.x));
            acc[dn_lo + q].im = fma2(dg, pk(sd.y, sd.w), pk(c_dn0 * pw, -sd.y));
        }
        if (!NORM && !active) continue;
        float nrm = 0.f;
        if (!NORM || active) {
            const float2 *sLs = sL + ls * LSTRIDE;
            const float fs = DAG ? 1.f : -1.f;  // sig of the forward hops
            hop2<0, false>(acc, pa, sLs + 0 * 10, fs);  ldrow<LS>(pa, in + nb(1, true));
            hop2<0, true>(acc, pb, sLs + 4 * 10, -fs);  ldrow<LS>(pb, in + nb(1, false));
            hop2<1, false>(acc, pa, sLs + 1 * 10, fs);  ldrow<LS>(pa, in + nb(2, true));
            hop2<1, true>(acc, pb, sLs + 5 * 10, -fs);  ldrow<LS>(pb, in + nb(2, false));
            hop2<2, false>(acc, pa, sLs + 2 * 10, fs);  ldrow<LS>(pa, in + nb(3, true));
            hop2<2, true>(acc, pb, sLs + 6 * 10, -fs);  ldrow<LS>(pb, in + nb(3, false));
            hop2<3, false>(acc, pa, sLs + 3 * 10, fs);
            if (EPI >= 2) {
                const float2 *zp = zu.zin + (size_t)rhs * (size_t)field + self_off;
#pragma unroll
                for (int k = 0; k < 12; ++k) pa[k] = ld_hint(reinterpret_cast<const float4 *>(zp + k * LS), l2_policy(zu.stream));
            }
            hop2<3, true>(acc, pb, sLs + 7 * 10, -fs);
            // (>= where == would do: the plain kernels spill 16 bytes instead of 32, 428 -> 412 us)
            if (rhs + 1 >= r1) pdl_dependents();
            float2 *o = out + self_off;
            float a = 1.f;
            if (EPI == 2 || EPI == 4) {
                const double ww = zu.ww[(size_t)rhs * zu.stride];
                a = ww > 0.0 ? (float)(zu.zz[(size_t)rhs * zu.stride] / ww) : 0.f;
            }
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                float2 re = unpk(acc[k].re), im = unpk(acc[k].im);
                if (EPI == 2 || EPI == 3) {
                    re = make_float2(fmaf(-a, re.x, pa[k].x), fmaf(-a, re.y, pa[k].z));
                    im = make_float2(fmaf(-a, im.x, pa[k].y), fmaf(-a, im.y, pa[k].w));
                } else if (EPI == 4) {
                    re = make_float2(fmaf(a, pa[k].x, re.x), fmaf(a, pa[k].z, re.y));
                    im = make_float2(fmaf(a, pa[k].y, im.x), fmaf(a, pa[k].w, im.y));
                }
                const float4 v = make_float4(re.x, im.x, re.y, im.y);
                if (EPI >= 2) st_hint(reinterpret_cast<float4 *>(o + k * LS), v, l2_policy(zu.stream));
                else *reinterpret_cast<float4 *>(o + k * LS) = v;
                if (NORM) nrm += re.x * re.x + im.x * im.x + re.y * re.y + im.y * im.y;
            }
            if (EPI >= 2 && rhs + 1 < r1) request_z(rhs + 1);
        }
        if (NORM) {
            __shared__ double wsum[33];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) nrm += __shfl_down_sync(0xffffffffu, nrm, o);
            norm_epilogue(nout, rhs, (double)nrm, wsum);
        }
    }
}

}  // namespace

// CTAs of 64 threads, 8 per SM (minb = 8, the default) or of 128, 4 per SM
// (minb = 4); 128 registers either way.
template <int LS>
void dslash_pair_ls(dwf_ctx *c, float2 *out, const float2 *in, bool dag, int nrhs, int minb, double *nslot, int nstride,
                    const ZUpdate *zu) {
    const Geom &g = c->g;
    constexpr int SPW = 32 / (LS / 2);
    const int threads = minb == 4 ? 128 : 64;
    const int spb = threads / 32 * SPW;
    const Brick &bk = c->brick[minb == 4];
    // right-hand sides per CTA: two share the staged links unless that leaves
    // SMs idle in a grid of few waves (in units of one right-hand side's work,
    // staging the links counts about a quarter)
    const double slots = (double)c->sm_count * (minb == 4 ? 4 : 8);
    auto cost = [&](int n) {
        const double w = (double)bk.count * ((nrhs + n - 1) / n) / slots;
        return (w < 4.0 ? std::ceil(w) : w) * (0.25 + n);
    };
    int rb = nrhs > 1 && cost(2) <= cost(1) ? 2 : 1;
    // at the short fifth extents the links are a larger share of the work: four
    // where that still leaves three waves of CTAs (16^3 x 32 x 8, three fields:
    // 248 -> 216 us; x 4, twelve fields: 799 -> 761; at Ls 32 four lose 3 %)
    if (LS <= 8 && nrhs > 2 && (double)bk.count * ((nrhs + 3) / 4) / slots >= 3.0) rb = 4;
    DWF_REQUIRE(bk.count < ((int64_t)1 << 31), DWF_EINVAL, "paired Dslash: grid too large");
    dim3 grid((unsigned)bk.count, (unsigned)((nrhs + rb - 1) / rb));
    const size_t smem = (size_t)spb * LSTRIDE * sizeof(float2);
    const int64_t field = g.V * g.Ls * 12;
    const float diag = (float)(5.0 - c->M5), mf = (float)c->mf;
    const float2 *U = c->U32.as<float2>();
    const NormOut nout = nslot ? norm_out(c, grid, nrhs, nslot, nstride) : NormOut{};
    ZUpdate z = zu ? *zu : ZUpdate{nullptr, nullptr, nullptr, 0, 0, 0};
    // Fields that do not fit in L2 together: the second field and the output, each
    // touched once, leave it first, so that the rows shared by neighbouring CTAs
    // stay (V-cycle at 16^3 x 32 x 16, four sources: 22.5 -> 21.6 ms).  Fields that
    // fit are read again by the next kernel: there it costs 1 % (8^3 x 16 x 16).
    z.stream = 3 * (int64_t)nrhs * field * (int64_t)sizeof(float2) > c->l2_bytes;
#define PL(D, E)                                                                                                  \
    launch_after(dslash_pair_kernel<D, LS, E>, grid, dim3(threads), smem, c->stream, out, in, U, g, bk, diag, mf, \
                 field, nout, z, nrhs, rb)
    if (zu && !nslot) PL(false, 3);
    else if (zu && zu->add) PL(false, 4);
    else if (zu) PL(true, 2);
    else if (nslot && dag) PL(true, 1);
    else if (nslot) PL(false, 1);
    else if (dag) PL(true, 0);
    else PL(false, 0);
#undef PL
    DWF_CHECK_LAUNCH();
    if (nslot) norm_finish(c, nout, grid, nrhs);
}

}  // namespace dwf
