"""The setup's block kernels at the edges of their tiles: every Nvec, blocks of
less than one stage and of many, runs that are no multiple of a stage, one
coarse site, block extents of 1 (a face on both sides of one layer)."""
import numpy as np
import pytest

import test_gpu_mg as M

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [((4, 4, 4, 4), 8, 32, (2, 2, 2, 2)), ((8, 4, 4, 4), 16, 24, (4, 4, 4, 4)), ((4, 2, 4, 4), 6, 16, (4, 2, 4, 4)),
         ((3, 3, 4, 2), 4, 12, (3, 3, 2, 1)), ((4, 4, 2, 4), 5, 8, (2, 1, 2, 2)), ((4, 2, 6, 4), 3, 6, (2, 2, 3, 2)),
         ((2, 4, 2, 2), 2, 4, (1, 2, 1, 1)), ((2, 2, 2, 3), 2, 2, (1, 1, 1, 1))]


@pytest.fixture(scope="module")
def G():
    from paper_1205_2933_gb300 import dwfmg
    return dwfmg


@pytest.mark.parametrize("dims,Ls,nvec,block", CASES)
@pytest.mark.parametrize("prec", [0, 1], ids=["f64", "f32"])
def test_basis_and_stencil(G, dims, Ls, nvec, block, prec):
    """Gamma split, block Gram-Schmidt and R D P of given vectors against the oracle's."""
    from gpu_util import to_canonical, rel_norm
    c = M.Case(G, dims=dims, Ls=Ls, mf=0.1, nvec=[nvec], block=[block], setup_iters0=0, setup_sweeps=0,
               smoother_prec=prec, coarse_prec=[prec])
    tol = 1e-12 if prec == 0 else 5e-6  # FP32: rounding of the basis through well-conditioned block triangles
    q = torch.empty(c.ctx.field_elems * nvec, dtype=torch.complex128, device="cuda")
    G.mg_get_vectors(c.ctx.h, 0, q)
    got = to_canonical(c.ctx, q, (nvec,) + c.op.shape, nrhs=nvec)
    ref = np.stack([c.mg.levels[0].transfer.vector(k) for k in range(nvec)])
    assert rel_norm(got, ref) < tol
    Y = c.mg.levels[1].op.Y
    y = torch.empty(Y.size, dtype=torch.complex128, device="cuda")
    G.mg_get_coarse_links(c.ctx.h, 1, y)
    assert rel_norm(y.cpu().numpy().reshape(Y.shape), Y) < tol
    c.close()
