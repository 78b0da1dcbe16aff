"""Rounding of the FP32 and FP64 paths against 64 bits: the bounds are what the
plainest kernel of the same sum leaves, with the spread between inputs."""
import numpy as np
import pytest

import paper_1205_2933_gb300.inputs as I
import test_gpu_mg as M

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def G():
    from paper_1205_2933_gb300 import dwfmg
    return dwfmg


def _ctx(dims, Ls):
    from gpu_util import ctx_for
    return ctx_for(I.epsilon_links(dims, 0.5, 1), dims, Ls, 1.8, 0.1)


def _randn(n, seed, dtype=torch.complex128):
    g = torch.Generator("cuda").manual_seed(seed)
    return torch.randn(n, dtype=torch.complex128, device="cuda", generator=g).to(dtype)


def _rel(a, b):
    return ((a.to(torch.complex128) - b).norm() / b.norm()).item()


@pytest.mark.parametrize("dag", [False, True])
@pytest.mark.parametrize("Ls", [4, 6, 8, 10, 12, 14, 16, 20, 24, 32, 48, 64])
def test_fp32_dslash(G, Ls, dag):
    """8.0e-8 at every fifth extent, whichever kernel takes it (one fifth of a
    percent between inputs; 2 % allowed)."""
    ctx = _ctx((8, 6, 8, 6), Ls)
    f = _randn(ctx.field_elems, 3, torch.complex64)
    out, ref = torch.empty_like(f), torch.empty(f.numel(), dtype=torch.complex128, device="cuda")
    G.dwf_apply(ctx.h, out, f, G.DWF_F32, dag, 1)
    G.dwf_apply(ctx.h, ref, f.to(torch.complex128), G.DWF_F64, dag, 1)
    assert _rel(out, ref) < 8.16e-8
    ctx.close()


@pytest.mark.parametrize("dims,Ls,nu,nrhs,bound",
                         [((8, 8, 8, 8), 4, 8, 1, 1.6e-7), ((8, 8, 8, 8), 8, 16, 1, 1.6e-7), ((8, 8, 8, 8), 16, 16, 1, 1.6e-7),
                          ((8, 6, 4, 8), 12, 16, 1, 1.6e-7), ((8, 6, 4, 8), 6, 8, 3, 1.6e-7), ((8, 6, 4, 8), 12, 16, 3, 1.6e-7),
                          ((8, 6, 4, 8), 20, 16, 3, 1.6e-7), ((8, 8, 8, 8), 8, 16, 3, 4.5e-7)])
def test_fp32_vcycle(G, dims, Ls, nu, nrhs, bound):
    """The V-cycle against the FP64 one, coarse iterations fixed: the smoother
    that keeps r leaves 1.3e-7, the one that carries z 3.7e-7 (which only batches
    use, and only where Ls / 2 divides 32); each with a fifth more."""
    out = []
    for prec in (G.DWF_F64, G.DWF_F32):
        ctx = _ctx(dims, Ls)
        p = M._params(G, setup_iters0=0, setup_sweeps=0, smoother_prec=prec, coarse_prec=[prec], coarsest_tol=0.0,
                      coarsest_maxiter=8, nu_post=nu)
        G.mg_setup(ctx.h, 2, [8], [(2, 2, 2, 2)], p, torch.from_numpy(I.random_vectors(4, dims, Ls, 3)).cuda())
        b = _randn(nrhs * ctx.field_elems, 5)
        out.append(torch.empty_like(b))
        G.mg_vcycle_batch(ctx.h, out[-1], b, nrhs)
        torch.cuda.synchronize()
        ctx.close()
    assert _rel(out[1], out[0]) < bound


def _gcr64(Y, dims, b, its, restart):
    """GCR of the coarse stencil Y [V][9][n][n] in FP64, its directions orthogonalised twice."""
    V, n = Y.shape[0], Y.shape[2]
    site = torch.arange(V, device="cuda").reshape(tuple(dims)[::-1])
    nb = [site.reshape(-1)]
    for mu in range(4):
        nb += [torch.roll(site, s, 3 - mu).reshape(-1) for s in (-1, 1)]

    def A(v):
        v = v.reshape(V, n)
        return sum(torch.einsum("skl,sl->sk", Y[:, d], v[nb[d]]) for d in range(9)).reshape(-1)

    x, r, Z, W = torch.zeros_like(b), b.clone(), [], []
    for _ in range(its):
        z, w = r.clone(), A(r)
        for zi, wi in 2 * list(zip(Z, W)):
            c = torch.vdot(wi, w)
            w, z = w - c * wi, z - c * zi
        nw = w.norm()
        Z.append(z / nw)
        W.append(w / nw)
        a = torch.vdot(W[-1], r)
        x, r = x + a * Z[-1], r - a * W[-1]
        if len(Z) == restart:
            r, Z, W = b - A(x), [], []
    return x


@pytest.mark.parametrize("prec", [0, 1], ids=["f64", "f32"])
@pytest.mark.parametrize("dims,Ls,nvec,block,restart,its,f32,f64",
                         [((8, 8, 8, 8), 4, 8, (2, 2, 2, 2), 16, 12, 1.36, 3.3), ((8, 8, 8, 8), 4, 16, (2, 2, 2, 2), 16, 32, 1.53, 4.1),
                          ((6, 6, 3, 6), 4, 24, (1, 1, 1, 1), 16, 16, 1.37, 3.6),
                          ((8, 8, 8, 8), 8, 24, (4, 4, 2, 2), 16, 24, 1.44, 3.8)])
def test_coarsest_gcr(G, dims, Ls, nvec, block, restart, its, f32, f64, prec):
    """A fixed number of coarsest GCR iterations against FP64 on the same links.
    f32 (1e-7), f64 (1e-16): what the solver with FP64 sums, two projections each
    and warp-wide stencil sums leaves; 15 % between one shape's right-hand sides."""
    ctx = _ctx(dims, Ls)
    p = M._params(G, setup_iters0=30, setup_sweeps=0, smoother_prec=prec, coarse_prec=[prec], coarsest_tol=0.0,
                  coarsest_maxiter=its, coarse_restart=restart)
    G.mg_setup(ctx.h, 2, [nvec], [block], p, torch.from_numpy(I.random_vectors(nvec // 2, dims, Ls, 3)).cuda())
    d, n = G.mg_level_info(ctx.h, 1)
    V, dt = int(np.prod(d)), torch.complex64 if prec else torch.complex128
    y = torch.empty(V * 9 * n * n, dtype=torch.complex128, device="cuda")
    G.mg_get_coarse_links(ctx.h, 1, y)
    Y = y.to(dt).to(torch.complex128).reshape(V, 9, n, n)
    err = 0.0
    for s in range(4):
        b = _randn(V * n, 7 + s, dt)
        x = torch.empty_like(b)
        G.mg_coarse_solve(ctx.h, 1, x, b)
        err += _rel(x, _gcr64(Y, d, b.to(torch.complex128), its, restart)) / 4
    assert err < 1.15 * (f32 * 1e-7 if prec else f64 * 1e-16)
    ctx.close()


@pytest.mark.parametrize("dims,Ls,nvec,block,restrict,prolong",
                         [((8, 8, 8, 8), 8, 8, (2, 2, 2, 2), 1.00, 0.63), ((8, 8, 8, 8), 4, 16, (2, 2, 2, 2), 0.95, 0.82),
                          ((8, 8, 8, 8), 16, 24, (4, 4, 4, 4), 2.7, 0.98), ((6, 6, 4, 8), 12, 32, (3, 3, 2, 4), 1.49, 1.11)])
def test_fp32_transfers(G, dims, Ls, nvec, block, restrict, prolong):
    """One restriction and one prolongation against FP64 on the same basis: what
    sums of whole products leave (1e-7), 4 % between inputs."""
    ctx = _ctx(dims, Ls)
    p = M._params(G, setup_iters0=4, setup_sweeps=0, smoother_prec=1, coarse_prec=[1])
    G.mg_setup(ctx.h, 2, [nvec], [block], p, torch.from_numpy(I.random_vectors(nvec // 2, dims, Ls, 3)).cuda())
    N = ctx.field_elems
    Q = torch.empty(nvec * N, dtype=torch.complex128, device="cuda")
    G.mg_get_vectors(ctx.h, 0, Q)
    torch.cuda.synchronize()
    Q = Q.reshape(nvec, N)
    d, n = G.mg_level_info(ctx.h, 1)
    site, xc, m = torch.arange(int(np.prod(dims)), device="cuda"), 0, 1
    for mu in range(4):
        xc = xc + (site % dims[mu] // block[mu]) * m
        site, m = site // dims[mu], m * d[mu]
    xc = xc.repeat_interleave(12 * Ls)  # the block of every element
    err = np.zeros(2)
    for s in range(4):
        f, out = _randn(N, 5 + s, torch.complex64).to(torch.complex128), torch.empty(m * n, dtype=torch.complex128, device="cuda")
        G.mg_restrict(ctx.h, 0, out, f)
        ref = torch.zeros(n, m, dtype=torch.complex128, device="cuda").index_add_(1, xc, Q.conj() * f)
        err[0] += _rel(out, ref.T.reshape(-1)) / 4
        c, out = _randn(m * n, 50 + s, torch.complex64).to(torch.complex128), torch.empty(N, dtype=torch.complex128, device="cuda")
        G.mg_prolong(ctx.h, 0, out, c)
        err[1] += _rel(out, (Q * c.reshape(m, n).T[:, xc]).sum(0)) / 4
    assert err[0] < 1.04e-7 * restrict and err[1] < 1.04e-7 * prolong
    ctx.close()


@pytest.mark.parametrize("dag", [False, True])
@pytest.mark.parametrize("prec", [0, 1], ids=["f64", "f32"])
@pytest.mark.parametrize("dims,Ls,nvec,block,f32,f64", [((8, 8, 8, 8), 8, 8, (2, 2, 2, 2), 2.12, 4.2),
                                                        ((8, 8, 8, 8), 8, 24, (4, 4, 2, 2), 3.57, 6.9),
                                                        ((8, 8, 8, 8), 4, 32, (2, 2, 2, 2), 4.11, 7.9)])
def test_coarse_operator(G, dims, Ls, nvec, block, f32, f64, prec, dag):
    """The coarse stencil, D and D^+, against FP64 on the same links: what one
    chain of whole products over all 9 Nvec links leaves (f32 1e-7, f64 1e-16;
    the latter with the reference's own)."""
    ctx = _ctx(dims, Ls)
    p = M._params(G, setup_iters0=4, setup_sweeps=0, smoother_prec=prec, coarse_prec=[prec])
    G.mg_setup(ctx.h, 2, [nvec], [block], p, torch.from_numpy(I.random_vectors(nvec // 2, dims, Ls, 3)).cuda())
    d, n = G.mg_level_info(ctx.h, 1)
    V, dt = int(np.prod(d)), torch.complex64 if prec else torch.complex128
    y = torch.empty(V * 9 * n * n, dtype=torch.complex128, device="cuda")
    G.mg_get_coarse_links(ctx.h, 1, y)
    Y = y.to(dt).to(torch.complex128).reshape(V, 9, n, n)
    site = torch.arange(V, device="cuda").reshape(tuple(d)[::-1])
    nb = [site.reshape(-1)]
    for mu in range(4):
        nb += [torch.roll(site, s, 3 - mu).reshape(-1) for s in (-1, 1)]
    err = 0.0
    for s in range(4):
        b = _randn(V * n, 7 + s, dt)
        out, v = torch.empty_like(b), b.to(torch.complex128).reshape(V, n)
        G.mg_coarse_apply(ctx.h, 1, out, b, dagger=dag, prec=prec)
        if dag:  # D^+ v at x: Y_d(y)^+ v(y) of the sites y whose direction d leads to x
            ref = torch.zeros_like(v)
            for k in range(9):
                ref.index_add_(0, nb[k], torch.einsum("slk,sl->sk", Y[:, k].conj(), v))
        else:
            ref = sum(torch.einsum("skl,sl->sk", Y[:, k], v[nb[k]]) for k in range(9))
        err += _rel(out, ref.reshape(-1)) / 4
    assert err < 1.05 * (f32 * 1e-7 if prec else f64 * 1e-16)
    ctx.close()


def test_network_forward(G):
    """The FP32 network (48 channels, three layers) against the FP64 oracle: 7.5e-7
    with sums of whole products, a tenth more allowed."""
    import test_gpu_net as T
    from oracle import net as N
    shape = N.NetShape(c_in=8, hidden=48, layers=3, nout=6, Ls=8)
    U = I.epsilon_links(T.DIMS, 0.3, 1)
    c = T.NetCase(G, U, shape)
    h0 = T._input(shape, T.DIMS, 20)
    ref, _ = N.forward(shape, c.p, U, h0, T.DIMS)
    out = c.forward(h0=h0)
    assert np.linalg.norm(out.reshape(-1) - ref.reshape(-1)) < 8.2e-7 * np.linalg.norm(ref)
    c.close()
