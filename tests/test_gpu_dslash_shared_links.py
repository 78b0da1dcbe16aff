"""The paired FP32 Dslash where a CTA applies its staged links to two or four
right-hand sides in turn, with an odd number of them (the last CTAs have fewer):
D and D^+ field by field, and every fused epilogue through the batched V-cycle
(norms added by the last CTA or by a launch of their own, the second field asked
for ahead, outputs that leave L2 first in fields larger than it)."""
import math

import numpy as np
import pytest

import paper_1205_2933_gb300.inputs as I
import test_gpu_mg as M

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# dims, Ls, right-hand sides, right-hand sides per CTA, CTAs whose norms the last one adds
CASES = [((8, 8, 4, 8), 16, 5, 2, True), ((8, 8, 8, 8), 16, 3, 2, False), ((12, 12, 12, 16), 16, 11, 2, False),
         ((6, 10, 6, 14), 12, 3, 2, False), ((16, 16, 8, 16), 8, 5, 4, False), ((16, 16, 16, 16), 4, 7, 4, False)]


def _per_cta(dims, Ls, nrhs):
    """The launch rule, restated for lattices that whole bricks cover."""
    slots = torch.cuda.get_device_properties(0).multi_processor_count * 8
    bricks = math.prod(dims) // (2 * (32 // (Ls // 2)))

    def cost(n):
        w = bricks * math.ceil(nrhs / n) / slots
        return (math.ceil(w) if w < 4 else w) * (0.25 + n)

    if Ls <= 8 and nrhs > 2 and bricks * math.ceil(nrhs / 4) / slots >= 3:
        return bricks, 4
    return bricks, 2 if nrhs > 1 and cost(2) <= cost(1) else 1


@pytest.fixture(scope="module")
def G():
    from paper_1205_2933_gb300 import dwfmg
    return dwfmg


def _ctx(dims, Ls):
    from gpu_util import ctx_for
    return ctx_for(I.epsilon_links(dims, 0.4, 1), dims, Ls, 1.8, 0.1)


@pytest.mark.parametrize("dims,Ls,nrhs,rb,few", CASES)
def test_apply_field_by_field(G, dims, Ls, nrhs, rb, few):
    """Each field as when it is alone, bit for bit."""
    bricks, per = _per_cta(dims, Ls, nrhs)
    assert per == rb and (bricks <= 256) == few
    ctx = _ctx(dims, Ls)
    n = ctx.field_elems
    f = torch.randn(nrhs * n, dtype=torch.complex64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    out, one = torch.empty_like(f), torch.empty(n, dtype=f.dtype, device="cuda")
    for dag in (False, True):
        G.dwf_apply(ctx.h, out, f, G.DWF_F32, dag, nrhs)
        for r in range(nrhs):
            G.dwf_apply(ctx.h, one, f[r * n:(r + 1) * n].clone(), G.DWF_F32, dag, 1)
            assert torch.equal(out[r * n:(r + 1) * n], one)
    ctx.close()


@pytest.mark.parametrize("dims,Ls,nrhs,rb,few", CASES)
def test_vcycle_field_by_field(G, dims, Ls, nrhs, rb, few):
    """Each field of a batched V-cycle against the V-cycle of that field alone, to
    the rounding of 5 smoothing steps in either form (3e-7), thirty times that;
    the sources differ in size, so that another field's sums would show."""
    ctx = _ctx(dims, Ls)
    p = M._params(G, setup_iters0=8, setup_sweeps=0, smoother_prec=1, coarse_prec=[1], coarsest_tol=0.0,
                  coarsest_maxiter=4, nu_post=5)
    G.mg_setup(ctx.h, 2, [8], [(2, 2, 2, 2)], p)
    n = ctx.field_elems
    b = torch.randn(nrhs, n, dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    b *= torch.arange(1, nrhs + 1, device="cuda")[:, None]
    x, y = torch.empty_like(b), torch.empty(n, dtype=b.dtype, device="cuda")
    G.mg_vcycle_batch(ctx.h, x.view(-1), b.view(-1), nrhs)
    for r in range(nrhs):
        G.mg_vcycle(ctx.h, y, b[r])
        torch.cuda.synchronize()
        assert ((x[r] - y).norm() / y.norm()).item() < 1e-5, r
    ctx.close()


@pytest.mark.parametrize("Ls", [4, 6, 10, 12, 16, 20, 24, 32, 48, 64])
def test_carried_updates_of_cg(G, Ls):
    """Eleven CG iterations, whose z and w the Dslash epilogues update, in FP32
    against FP64 (3e-7 per eight iterations at Ls 8, thirty times that)."""
    dims = (6, 4, 4, 6)
    ctx = _ctx(dims, Ls)
    b = torch.randn(ctx.field_elems, dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    x = [torch.zeros_like(b), torch.zeros_like(b)]
    for i in (0, 1):
        assert G.dwf_cg_solve(ctx.h, b, x[i], 1e-14, 11, 1, i, check=False).iters == 11
    assert ((x[1] - x[0]).norm() / x[0].norm()).item() < 1e-5
    ctx.close()
