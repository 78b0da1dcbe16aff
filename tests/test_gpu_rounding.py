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
