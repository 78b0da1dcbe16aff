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
