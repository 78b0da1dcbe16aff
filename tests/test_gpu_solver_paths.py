"""The solver paths chosen by a size, a type or a count, each at the edges of
its rule: the coarsest GCR with its vectors in shared memory or not, the FP32
CG in chunks, the FP64 V-cycle in the fused form, one right-hand side through
the batched solver, and setups that take over the buffers of an earlier one."""
import numpy as np
import pytest

import oracle
from oracle import mg as OM
import paper_1205_2933_gb300.inputs as I
import test_gpu_mg as M

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def G():
    from paper_1205_2933_gb300 import dwfmg
    return dwfmg


def _setup(G, ctx, nvec, block, seed=3, **kw):
    p = M._params(G, **kw)
    start = torch.from_numpy(I.random_vectors(nvec // 2, ctx.dims, ctx.Ls, seed)).cuda()
    G.mg_setup(ctx.h, 2, [nvec], [block], p, start)
    return p


def _ctx(dims, Ls, mf=0.1):
    from gpu_util import ctx_for
    ctx = ctx_for(I.epsilon_links(dims, 0.3, 1), dims, Ls, 1.8, mf)
    ctx.dims, ctx.Ls = dims, Ls
    return ctx


# One coarse site; 24 sites, links cached; 648 sites, 5 to a CTA and 3 in the
# last, links cached or not; 2048 sites of 32 components, whose 34 FP64
# vectors do not fit a CTA's shared memory (FP32 ones do); the 33-point stencil.
COARSE = [((2, 2, 2, 2), 2, 2, (2, 2, 2, 2), 16, 0), ((6, 4, 4, 4), 4, 24, (2, 2, 2, 2), 8, 0),
          ((6, 6, 3, 6), 4, 6, (1, 1, 1, 1), 16, 0), ((6, 6, 3, 6), 4, 24, (1, 1, 1, 1), 5, 0),
          ((8, 8, 8, 4), 4, 32, (1, 1, 1, 1), 16, 0), ((4, 6, 4, 4), 4, 8, (2, 2, 2, 2), 16, 1)]


@pytest.mark.parametrize("dims,Ls,nvec,block,restart,squared", COARSE)
@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
def test_coarsest_gcr_step_for_step(G, dims, Ls, nvec, block, restart, squared, prec):
    """A fixed number of GCR iterations equals the oracle's GCR on the same
    stencil (applied by mg_coarse_apply): FP64 to 1e-9, FP32 arithmetic (FP32 or
    BF16 links) to 1e-4, its unit roundoff times 20 iterations times a
    condition of a hundred."""
    sp, cp = {"f64": (0, 0), "f32": (1, G.DWF_F32), "bf16": (1, G.DWF_BF16)}[prec]
    ctx = _ctx(dims, Ls)
    its = min(20, nvec // 2)
    _setup(G, ctx, nvec, block, setup_iters0=0, setup_sweeps=0, smoother_prec=sp, coarse_prec=[cp], coarsen=squared,
           coarsest_tol=0.0, coarsest_maxiter=its, coarse_restart=restart)
    d, n = G.mg_level_info(ctx.h, 1)
    dt = torch.complex128 if sp == 0 else torch.complex64
    b = torch.from_numpy(I.gauss_complex((int(np.prod(d)) * n,), 33, 50)).to(dt).cuda()
    x = torch.empty_like(b)
    G.mg_coarse_solve(ctx.h, 1, x, b)

    def apply(v):
        vt = torch.from_numpy(np.ascontiguousarray(v)).to(dt).cuda()
        out = torch.empty_like(vt)
        G.mg_coarse_apply(ctx.h, 1, out, vt, prec=sp)
        return out.cpu().numpy().astype(np.complex128)

    ref, _ = OM.gcr(apply, b.cpu().numpy().astype(np.complex128), tol=0.0, maxiter=its, restart=restart)
    assert np.linalg.norm(x.cpu().numpy() - ref) / np.linalg.norm(ref) < (1e-9 if sp == 0 else 1e-4)
    ctx.close()


@pytest.mark.parametrize("maxiter", [1, 7, 8, 9, 16, 21])
@pytest.mark.parametrize("Ls", [8, 3, 12], ids=["Ls8", "Ls3", "Ls12"])
def test_fp32_cg_iterations(G, Ls, maxiter):
    """dwf_cg_solve stops at maxiter whatever the chunk, from a guess; its x is
    the oracle's CGNR iterate to FP32 rounding (two members, one a multiple)."""
    from gpu_util import to_internal, to_canonical, rel_norm
    dims = (4, 4, 2, 4)
    ctx = _ctx(dims, Ls)
    op = OM.FineOp(oracle.DWF(I.epsilon_links(dims, 0.3, 1), dims, Ls, 1.8, 0.1))
    b, x0 = I.gaussian_source(dims, Ls, 2), 0.1 * I.gaussian_source(dims, Ls, 3)
    bt, xt = (to_internal(ctx, np.stack([v, 2 * v]), nrhs=2) for v in (b, x0))
    st = G.dwf_cg_solve(ctx.h, bt, xt, 1e-14, maxiter, 2, G.DWF_F32, check=False)
    assert st.iters == 2 * maxiter
    got = to_canonical(ctx, xt, (2,) + b.shape, nrhs=2)
    ref, _ = OM.cgnr(op.apply, op.apply_dag, b.reshape(op.shape), tol=0.0, maxiter=maxiter, x0=x0.reshape(op.shape))
    for k in (0, 1):
        assert rel_norm(got[k] / (k + 1), ref.reshape(b.shape)) < 1e-4
    ctx.close()


@pytest.mark.parametrize("cfg,nu", [(M.SMALL, 1), (M.SMALL, 8), (M.RAGGED, 5)])
def test_fp64_vcycle(G, cfg, nu):
    """The FP64 V-cycle at several smoother lengths against the oracle's."""
    from gpu_util import to_internal, to_canonical, rel_norm
    c = M.Case(G, **cfg, setup_iters0=4, setup_sweeps=0, coarsest_tol=0.0, coarsest_maxiter=6, nu_post=nu)
    b = I.gaussian_source(c.dims, c.Ls, 31)
    bt = to_internal(c.ctx, b)
    xt = torch.empty_like(bt)
    G.mg_vcycle(c.ctx.h, xt, bt)
    ref = c.mg.vcycle(0, b.reshape(c.op.shape)).reshape(b.shape)
    assert rel_norm(to_canonical(c.ctx, xt, b.shape), ref) < 1e-9
    c.close()


@pytest.mark.parametrize("prec,tol", [(0, 1e-9), (1, 1e-4)], ids=["f64", "f32"])
@pytest.mark.parametrize("dims,Ls", [((8, 8, 8, 8), 8), ((6, 4, 4, 4), 6)], ids=["many-ctas", "few-ctas"])
def test_smoother_forms_agree(G, dims, Ls, prec, tol, monkeypatch):
    """The V-cycle with the norms summed by the last CTA (few CTAs) and by a
    launch of their own (many), against the launch-by-launch smoother."""
    x = []
    for form in ("1", "0"):
        monkeypatch.setenv("DWF_SMOOTHER_HISTORY", form)
        ctx = _ctx(dims, Ls)
        _setup(G, ctx, 8, (2, 2, 2, 2), setup_iters0=0, setup_sweeps=0, smoother_prec=prec, coarse_prec=[prec],
               coarsest_tol=0.0, coarsest_maxiter=4)
        b = torch.from_numpy(I.gaussian_source(dims, Ls, 5).reshape(-1)).cuda()
        x.append(torch.empty_like(b))
        G.mg_vcycle(ctx.h, x[-1], b)
        torch.cuda.synchronize()
        ctx.close()
    assert ((x[0] - x[1]).norm() / x[1].norm()).item() < tol


@pytest.mark.parametrize("maxiter", [1, 3, 4, 9])
@pytest.mark.parametrize("prec", [0, 1], ids=["f64", "f32"])
def test_single_solve_stops_at_outer_maxiter(G, prec, maxiter):
    ctx = _ctx((4, 4, 4, 4), 8)
    _setup(G, ctx, 8, (2, 2, 2, 2), setup_iters0=0, setup_sweeps=0, smoother_prec=prec, coarse_prec=[prec],
           outer_maxiter=maxiter, outer_restart=4)
    b = torch.from_numpy(I.gaussian_source((4, 4, 4, 4), 8, 5).reshape(-1)).cuda()
    x = torch.zeros_like(b)
    st = G.mg_solve(ctx.h, b, x, 1e-15, check=False)
    assert st.iters == maxiter and 0.0 < st.true_res < 1.0
    ctx.close()


@pytest.mark.parametrize("prec,tol", [(0, 1e-12), (1, 1e-5)], ids=["f64", "f32"])
def test_setup_after_setup(G, prec, tol):
    """A setup on a context that has one (larger, smaller, of the same size)
    gives what a fresh context gives."""
    def links(ctx, nvec, block):
        _setup(G, ctx, nvec, block, setup_iters0=8, setup_sweeps=1, smoother_prec=prec, coarse_prec=[prec])
        d, n = G.mg_level_info(ctx.h, 1)
        y = torch.empty(int(np.prod(d)) * 9 * n * n, dtype=torch.complex128, device="cuda")
        G.mg_get_coarse_links(ctx.h, 1, y)
        b = torch.from_numpy(I.gaussian_source(ctx.dims, ctx.Ls, 5).reshape(-1)).cuda()
        x = torch.empty_like(b)
        G.mg_vcycle(ctx.h, x, b)
        torch.cuda.synchronize()
        return y, x

    old = _ctx((4, 4, 4, 4), 8)
    for nvec, block in [(8, (2, 2, 2, 2)), (8, (2, 2, 2, 2)), (16, (2, 2, 2, 2)), (8, (4, 2, 2, 2)), (8, (2, 2, 2, 2))]:
        new = _ctx((4, 4, 4, 4), 8)
        for a, b in zip(links(old, nvec, block), links(new, nvec, block)):
            assert ((a - b).norm() / b.norm()).item() < tol
        new.close()
    old.close()


def test_coarse_shapes_of_a_batch_share_a_kernel(G):
    """Lattices of one context solve from threads of their own, with the same
    coarsest kernel at different shared-memory needs: one's launch must not
    lower what another's may ask for."""
    dims = [(8, 8, 8, 8), (4, 4, 4, 4), (4, 4, 4, 8)]
    bc = G.BatchContext(dims, 4, 1.8, 0.1, [torch.from_numpy(I.epsilon_links(d, 0.3, 1)).cuda() for d in dims])
    p = M._params(G, setup_iters0=16, smoother_prec=1, coarse_prec=[1])
    G.mg_setup(bc.h, 2, [8], [(2, 2, 2, 2)], p)
    b = torch.from_numpy(np.concatenate([I.gaussian_source(d, 4, 5).reshape(-1) for d in dims])).cuda()
    for _ in range(10):
        x = torch.zeros_like(b)
        assert G.mg_solve(bc.h, b, x, 1e-8).true_res <= 1e-8
    bc.close()


@pytest.mark.parametrize("Ls,nrhs", [(8, 3), (4, 5)])
def test_apply_of_several_fields_per_link(G, Ls, nrhs):
    """Large grids at short fifth extents: each field as when it is alone, bit for bit."""
    ctx = _ctx((16, 16, 16, 32), Ls)
    n = ctx.field_elems
    f = torch.randn(nrhs * n, dtype=torch.complex64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    out, one = torch.empty_like(f), torch.empty(n, dtype=f.dtype, device="cuda")
    G.dwf_apply(ctx.h, out, f, G.DWF_F32, False, nrhs)
    for r in range(nrhs):
        G.dwf_apply(ctx.h, one, f[r * n:(r + 1) * n].clone(), G.DWF_F32, False, 1)
        assert torch.equal(out[r * n:(r + 1) * n], one)
    ctx.close()
