"""Restriction and prolongation at the edges of their tiles: runs that are no
multiple of a stage, blocks of one piece and of many (one coarse site included),
every Nvec, and the widths of the batched kernels (the register tiles' 1, 2, 4,
6, 8 and 12 right-hand sides, masked ones, several groups)."""
import numpy as np
import pytest

import paper_1205_2933_gb300.inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [((4, 2, 6, 4), 3, 6, (2, 2, 3, 2)), ((4, 4, 4, 4), 8, 32, (2, 2, 2, 2)), ((8, 4, 4, 4), 16, 24, (4, 4, 4, 4)),
         ((4, 4, 4, 4), 5, 16, (4, 4, 4, 4)), ((2, 2, 2, 3), 1, 2, (1, 1, 1, 1)), ((3, 3, 4, 2), 4, 12, (3, 3, 2, 1)),
         ((4, 4, 4, 8), 4, 8, (2, 2, 2, 2)), ((2, 4, 2, 2), 2, 4, (2, 1, 2, 2))]


@pytest.fixture(scope="module")
def G():
    from paper_1205_2933_gb300 import dwfmg
    return dwfmg


def _setup(G, dims, Ls, nvec, block, prec, **kw):
    from gpu_util import ctx_for
    ctx = ctx_for(I.epsilon_links(dims, 0.3, 1), dims, Ls, 1.8, 0.1)
    p = G.mg_default_params()
    p.setup_iters0, p.split, p.smoother_prec = 0, 0, prec
    p.coarse_prec[0] = prec
    for k, v in kw.items():
        setattr(p, k, v)
    start = I.random_vectors(nvec, dims, Ls, 3)
    G.mg_setup(ctx.h, 2, [nvec], [block], p, torch.from_numpy(start).cuda())
    n = ctx.field_elems
    q = torch.empty(nvec * n, dtype=torch.complex128, device="cuda")
    G.mg_get_vectors(ctx.h, 0, q)
    torch.cuda.synchronize()
    # (nvec, coarse site, elements of the block)
    X, Y, Z, T = dims
    x, y, z, t = block
    to_blocks = lambda f: (f.reshape(-1, T // t, t, Z // z, z, Y // y, y, X // x, x, 12 * Ls)
                           .transpose(0, 1, 3, 5, 7, 2, 4, 6, 8, 9).reshape(f.reshape(-1, n).shape[0], n // (12 * Ls * x * y * z * t), -1))
    return ctx, to_blocks, to_blocks(q.cpu().numpy())


@pytest.mark.parametrize("dims,Ls,nvec,block", CASES)
@pytest.mark.parametrize("prec", [0, 1], ids=["f64", "f32"])
def test_restrict_prolong(G, dims, Ls, nvec, block, prec):
    ctx, to_blocks, Q = _setup(G, dims, Ls, nvec, block, prec)
    n, Vc = ctx.field_elems, Q.shape[1]
    tol = 1e-13 if prec == 0 else 2e-6  # sums of at most 12,288 products, FP32: 2^-24 times a few
    f = torch.from_numpy(I.gauss_complex((n,), 21, 50)).cuda()
    c = torch.empty(Vc * nvec, dtype=torch.complex128, device="cuda")
    G.mg_restrict(ctx.h, 0, c, f)
    ref = np.einsum("kbi,bi->bk", Q.conj(), to_blocks(f.cpu().numpy())[0])
    got = c.cpu().numpy().reshape(Vc, nvec)
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
    cin = I.gauss_complex((Vc, nvec), 22, 50)
    fo = torch.empty(n, dtype=torch.complex128, device="cuda")
    G.mg_prolong(ctx.h, 0, fo, torch.from_numpy(cin.reshape(-1)).cuda())
    ref = np.einsum("kbi,bk->bi", Q, cin)
    assert np.linalg.norm(to_blocks(fo.cpu().numpy())[0] - ref) <= tol * np.linalg.norm(ref)
    ctx.close()


@pytest.mark.parametrize("dims,Ls,nvec,block", CASES)
@pytest.mark.parametrize("nrhs", [2, 3, 5, 7, 12, 13, 29])
def test_batched_transfers(G, dims, Ls, nvec, block, nrhs):
    """With one coarse GCR step and no smoothing the V-cycle is alpha P R b (a
    complex alpha for every right-hand side): x is parallel to Q Q^+ b."""
    ctx, to_blocks, Q = _setup(G, dims, Ls, nvec, block, 1, nu_post=0, coarsest_tol=0.0, coarsest_maxiter=1)
    n = ctx.field_elems
    b = torch.from_numpy(I.gauss_complex((nrhs * n,), 23, 50)).cuda()
    x = torch.empty_like(b)
    G.mg_vcycle_batch(ctx.h, x, b, nrhs)
    bb = to_blocks(b.cpu().numpy())
    ref = np.einsum("kbi,rbk->rbi", Q, np.einsum("kbi,rbi->rbk", Q.conj(), bb)).reshape(nrhs, -1)
    got = to_blocks(x.cpu().numpy()).reshape(nrhs, -1)
    al = np.einsum("ri,ri->r", ref.conj(), got) / np.einsum("ri,ri->r", ref.conj(), ref)
    assert np.all(np.abs(al) > 0)
    off = np.linalg.norm(got - al[:, None] * ref, axis=1) / np.linalg.norm(got, axis=1)
    assert off.max() <= 4e-6, off  # two FP32 transfers and the coarse step
    ctx.close()
