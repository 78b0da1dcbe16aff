// Addressing of blocks of the finer lattice, shared by the transfer kernels and
// by the kernels of the setup, and the Nvec dispatch.
#pragma once

#include <algorithm>

#include "fastdiv.cuh"
#include "mg.cuh"

namespace dwf {

namespace {

// A box of finer sites (a block, or one face of it) taken in the order of its
// sites, each with its contiguous run of elements.
struct Box {
    int n[3];        // extents in x, y, z
    int L[3];        // finer lattice extents in x, y, z
    int run;
    FastDiv drun, dn[3];
};

Box make_box(const int n[4], const int L[4], int run) {
    Box b;
    b.run = run;
    b.drun = fast_div(run);
    for (int i = 0; i < 3; ++i) {
        b.n[i] = n[i];
        b.L[i] = L[i];
        b.dn[i] = fast_div(n[i]);
    }
    return b;
}

// address of element e of the box whose first site is `origin`
__device__ __forceinline__ int64_t box_elem(const Box &m, int64_t origin, unsigned e) {
    unsigned i = m.drun.div(e);
    const unsigned rem = e - i * m.run;
    unsigned q = m.dn[0].div(i);
    const unsigned o0 = i - q * m.n[0];
    i = q;
    q = m.dn[1].div(i);
    const unsigned o1 = i - q * m.n[1];
    i = q;
    q = m.dn[2].div(i);
    const unsigned o2 = i - q * m.n[2];
    return (origin + (((int64_t)q * m.L[2] + o2) * m.L[1] + o1) * m.L[0] + o0) * m.run + rem;
}

struct BlockMap {
    int L[4];        // finer lattice
    int b[4];        // block
    int Lc[4];       // coarse lattice
    int run;         // contiguous elements per finer site = ncomp * Ls
    int64_t bsites;  // sites per block
    int64_t nelem;   // elements per finer field
    Box box;         // the block's elements
};

// site index of the first finer site of block xc
__device__ __forceinline__ int64_t block_origin(const BlockMap &m, int64_t xc) {
    int64_t t = xc;
    const int c0 = (int)(t % m.Lc[0]); t /= m.Lc[0];
    const int c1 = (int)(t % m.Lc[1]); t /= m.Lc[1];
    const int c2 = (int)(t % m.Lc[2]), c3 = (int)(t / m.Lc[2]);
    return (((int64_t)c3 * m.b[3] * m.L[2] + c2 * m.b[2]) * m.L[1] + c1 * m.b[1]) * m.L[0] + c0 * m.b[0];
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
    m.box = make_box(m.b, m.L, m.run);
    return m;
}

int64_t ncoarse(const BlockMap &m) { return (int64_t)m.Lc[0] * m.Lc[1] * m.Lc[2] * m.Lc[3]; }

template <int BYTES> __device__ __forceinline__ void cp_async(void *dst, const void *src, bool on) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = on ? BYTES : 0;  // 0: the destination is filled with zeros
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(d), "l"(src), "n"(BYTES), "r"(n) : "memory");
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

}  // namespace dwf
