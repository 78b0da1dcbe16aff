"""The FP32 coarsest solve at any scale of its right-hand side: multiplying b
by a power of two multiplies x by the same, bit for bit."""
import numpy as np
import pytest

import paper_1205_2933_gb300.inputs as I
import test_gpu_mg as M

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# the last shape's 34 vectors of 41 sites do not fit a CTA's shared memory (the
# kernel of large problems) nor the static scratch
@pytest.mark.parametrize("dims,nvec,block,links,static",
                         [((4, 4, 4, 4), 8, (2, 2, 2, 2), 1, False), ((4, 4, 4, 4), 8, (2, 2, 2, 2), 1, True),
                          ((6, 6, 3, 6), 24, (1, 1, 1, 1), 2, False), ((6, 6, 3, 6), 24, (1, 1, 1, 1), 2, True),
                          ((12, 8, 8, 8), 32, (1, 1, 1, 1), 1, False)])
def test_scaled_right_hand_side(dims, nvec, block, links, static):
    from gpu_util import ctx_for
    from paper_1205_2933_gb300 import dwfmg as G
    ctx = ctx_for(I.epsilon_links(dims, 0.3, 1), dims, 4, 1.8, 0.1)
    # more iterations than one restart: the true residual is formed again
    p = M._params(G, setup_iters0=0, setup_sweeps=0, smoother_prec=1, coarse_prec=[links], coarsest_tol=1e-5,
                  coarsest_maxiter=24, coarse_restart=16 if nvec > 8 else 8)
    start = torch.from_numpy(I.random_vectors(nvec // 2, dims, 4, 3)).cuda()
    G.mg_setup(ctx.h, 2, [nvec], [block], p, start)
    d, n = G.mg_level_info(ctx.h, 1)
    solve = G.mg_coarse_solve_static if static else G.mg_coarse_solve
    N = int(np.prod(d)) * n
    b = torch.from_numpy(I.gauss_complex((N,), 33, 50)).to(torch.complex64).cuda()
    x = torch.empty_like(b)
    solve(ctx.h, 1, x, b)
    res = torch.empty_like(b)
    G.mg_coarse_apply(ctx.h, 1, res, x, prec=G.DWF_F32)
    assert (b - res).norm().item() < b.norm().item()
    for e in (-90, -75, -66, 62, 70, 100):
        y = torch.empty_like(b)
        solve(ctx.h, 1, y, b * 2.0 ** e)
        assert torch.equal(y, x * 2.0 ** e), e
    ctx.close()
