"""The paired FP32 Dslash at the edges of its bricks and warps: every fifth
extent it is instantiated for (idle lanes where Ls/2 does not divide 32),
extents that no brick divides, extents 1 and 2, several right-hand sides per
CTA, misaligned fields, and its fused epilogues at a fifth extent that is no
power of two."""
import numpy as np
import pytest

import oracle
import paper_1205_2933_gb300.inputs as I
import test_gpu_mg as M

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def G():
    from paper_1205_2933_gb300 import dwfmg
    return dwfmg


@pytest.mark.parametrize("dims,Ls", [((3, 5, 2, 7), 4), ((5, 3, 7, 1), 6), ((4, 4, 4, 6), 8), ((3, 1, 5, 4), 10),
                                     ((6, 5, 3, 2), 12), ((7, 3, 2, 3), 16), ((3, 3, 2, 5), 20), ((2, 5, 3, 3), 24),
                                     ((1, 4, 3, 3), 32), ((2, 3, 1, 5), 48), ((3, 2, 3, 2), 64), ((3, 2, 4, 2), 14)])
@pytest.mark.parametrize("nrhs", [1, 6])
def test_apply(G, dims, Ls, nrhs):
    from gpu_util import ctx_for, to_internal, to_canonical, rel_norm, rel_max
    U = I.epsilon_links(dims, 0.6, 1)
    ctx = ctx_for(U, dims, Ls, 1.8, 0.07)
    fs = np.stack([I.gaussian_source(dims, Ls, 5 + i) for i in range(nrhs)])
    t = to_internal(ctx, fs, G.DWF_F32, nrhs=nrhs)
    o = oracle.DWF(U, dims, Ls, 1.8, 0.07)
    for dag in (False, True):
        out = torch.full_like(t, float("nan"))
        G.dwf_apply(ctx.h, out, t, G.DWF_F32, dag, nrhs)
        got = to_canonical(ctx, out, fs.shape, G.DWF_F32, nrhs=nrhs)
        ref = np.stack([o.Ddag(f) if dag else o.D(f) for f in fs])
        assert rel_norm(got, ref) < 1e-6 and rel_max(got, ref) < 2e-6
        # fields that start 8 bytes off a 16-byte boundary give the same up to rounding
        buf = torch.empty(2 * t.numel() + 2, dtype=torch.complex64, device="cuda")
        a, b = buf[1:1 + t.numel()], buf[1 + t.numel():1 + 2 * t.numel()]
        a.copy_(t)
        G.dwf_apply(ctx.h, b, a, G.DWF_F32, dag, nrhs)
        assert ((b - out).norm() / out.norm()).item() < 5e-7
    ctx.close()


@pytest.mark.parametrize("dims,Ls,nu", [((6, 4, 2, 4), 12, 4), ((2, 6, 4, 4), 6, 5)])
def test_fused_epilogues(G, dims, Ls, nu):
    """The batched FP32 V-cycle (norms, b - D x, z - a D^+ w, D z + b w) against the oracle's."""
    from gpu_util import to_internal, to_canonical, rel_norm
    c = M.Case(G, dims=dims, Ls=Ls, mf=0.1, nvec=[8], block=[(2, 2, 2, 2)], setup_iters0=10, setup_sweeps=0,
               smoother_prec=G.DWF_F32, coarse_prec=[G.DWF_F32], coarsest_tol=0.0, coarsest_maxiter=8, nu_post=nu)
    nr = 5
    bs = [I.gaussian_source(c.dims, c.Ls, 40 + r) for r in range(nr)]
    bt = torch.cat([to_internal(c.ctx, b) for b in bs])
    xb = torch.empty_like(bt)
    G.mg_vcycle_batch(c.ctx.h, xb, bt, nr)
    n = c.ctx.field_elems
    for r in range(nr):
        got = to_canonical(c.ctx, xb[r * n:(r + 1) * n].contiguous(), bs[r].shape)
        ref = c.mg.vcycle(0, bs[r].reshape(c.op.shape)).reshape(bs[r].shape)
        assert rel_norm(got, ref) < 1e-4  # FP32 rounding through the relaxation, 8 coarse steps and nu smoothing steps
    c.close()
