"""Calls at the ends of what the library accepts: parameters above the limit of
a fused kernel, and what the statistics say of such calls."""
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


def _setup(G, dims=(4, 4, 4, 4), Ls=8, nvec=8, block=(2, 2, 2, 2), **kw):
    from gpu_util import ctx_for
    ctx = ctx_for(I.epsilon_links(dims, 0.3, 1), dims, Ls, 1.8, 0.1)
    p = M._params(G, **kw)
    start = torch.from_numpy(I.random_vectors(nvec // 2, dims, Ls, 3)).cuda()
    G.mg_setup(ctx.h, 2, [nvec], [block], p, start)
    return ctx


@pytest.mark.parametrize("prec", [0, 1], ids=["f64", "f32"])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_coarse_restart_beyond_the_fused_solver(G, prec, nrhs):
    """coarse_restart up to 64 is accepted; above 32 the coarsest solve runs
    launch by launch with host reads, which no graph may hold.  A solve of
    several V-cycles with the default parameters reaches its tolerance."""
    dims, Ls = (4, 4, 4, 4), 8
    ctx = _setup(G, dims, Ls, setup_iters0=8, setup_sweeps=0, smoother_prec=prec, coarse_prec=[prec], coarse_restart=40)
    b = np.concatenate([I.gaussian_source(dims, Ls, 5 + r).reshape(-1) for r in range(nrhs)])
    b = torch.from_numpy(b).cuda()
    x = torch.zeros_like(b)
    st = G.mg_solve(ctx.h, b, x, 1e-8, nrhs)
    assert st.true_res <= 1e-8 and st.iters > 2 * nrhs
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1], ids=["f64", "f32"])
@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("restart", [16, 40])
def test_coarse_applications_are_counted(G, prec, nrhs, restart):
    """Each outer iteration runs at least one coarsest iteration, by the fused
    solver or launch by launch: the statistics count them in both."""
    dims, Ls = (4, 4, 4, 4), 8
    ctx = _setup(G, dims, Ls, setup_iters0=8, setup_sweeps=0, smoother_prec=prec, coarse_prec=[prec],
                 coarse_restart=restart, graph=0, outer_maxiter=4, outer_restart=4)
    b = np.concatenate([I.gaussian_source(dims, Ls, 5 + r).reshape(-1) for r in range(nrhs)])
    b = torch.from_numpy(b).cuda()
    st = G.mg_solve(ctx.h, b, torch.zeros_like(b), 1e-14, nrhs, check=False)
    assert st.iters == 4 * nrhs and st.coarse_applies[1] >= st.iters
    ctx.close()


@pytest.mark.parametrize("where", ["host", "device"])
def test_start_vectors_off_a_16_byte_boundary(G, where):
    """Start vectors may lie at any 8-byte boundary, on the device as on the host."""
    from gpu_util import ctx_for
    dims, Ls, nvec = (4, 4, 4, 4), 4, 8
    start = I.random_vectors(nvec // 2, dims, Ls, 3).reshape(-1)
    if where == "device":
        buf = torch.empty(2 * start.size + 2, dtype=torch.float64, device="cuda")
        off = buf[1:1 + 2 * start.size]
        off.copy_(torch.from_numpy(start.view(np.float64)))
    else:
        buf = np.empty(2 * start.size + 2)
        off = buf[1:1 + 2 * start.size]
        off[:] = start.view(np.float64)
    q = []
    for s in (torch.from_numpy(start).cuda(), off):
        ctx = ctx_for(I.epsilon_links(dims, 0.3, 1), dims, Ls, 1.8, 0.1)
        G.mg_setup(ctx.h, 2, [nvec], [(2, 2, 2, 2)], M._params(G, setup_iters0=4, setup_sweeps=0), s)
        q.append(torch.empty(nvec * ctx.field_elems, dtype=torch.complex128, device="cuda"))
        G.mg_get_vectors(ctx.h, 0, q[-1])
        torch.cuda.synchronize()
        ctx.close()
    assert torch.equal(q[0], q[1])


SIDE = """
import numpy as np, torch
import paper_1205_2933_gb300.inputs as I
import test_gpu_mg as M
from paper_1205_2933_gb300 import dwfmg as G
from gpu_util import ctx_for
dims, Ls, nvec, nr = (8, 6, 4, 6), 4, 24, 4
ctx = ctx_for(I.epsilon_links(dims, 0.3, 1), dims, Ls, 1.8, 0.1)
p = M._params(G, setup_iters0=0, setup_sweeps=0, smoother_prec=1, coarse_prec=[1], coarsest_tol=0.0, coarsest_maxiter=12)
G.mg_setup(ctx.h, 2, [nvec], [(1, 1, 1, 1)], p, torch.from_numpy(I.random_vectors(nvec // 2, dims, Ls, 3)).cuda())
b = torch.cat([torch.from_numpy(I.gaussian_source(dims, Ls, 40 + r).reshape(-1)).cuda() for r in range(nr)])
x, y, n = torch.empty_like(b), torch.empty_like(b), ctx.field_elems
G.mg_vcycle_batch(ctx.h, x, b, nr)
for r in range(nr):
    G.mg_vcycle(ctx.h, y[r * n:(r + 1) * n], b[r * n:(r + 1) * n])
torch.cuda.synchronize()
print("err", ((x - y).norm() / y.norm()).item())
"""


def test_coarsest_solves_side_by_side():
    """Three coarsest solves at a time, each on a third of the SMs, where a
    third of them cannot hold the vectors (1152 sites x 24, 34 vectors): as one
    solve at a time to FP32 rounding (12 coarsest iterations, 8 smoothing steps)."""
    import os
    import subprocess
    import sys
    here = os.path.dirname(os.path.abspath(__file__))
    env = dict(os.environ, DWF_COARSE_BATCH="0", PYTHONPATH=os.pathsep.join([os.path.dirname(here), here]))
    out = subprocess.run([sys.executable, "-c", SIDE], env=env, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    assert float(out.stdout.split()[-1]) < 1e-4
