"""The FP32 relaxation of the setup's start vectors keeps, at every fifth extent,
the form whose rounding it had: within twice what eight FP32 CGNR steps with a
fresh z = D^+ r leave (1.3e-6 at Ls 12) or with a carried z (3.4e-6 at Ls 4, 8,
16), against the FP64 library on the same vectors."""
import pytest

import paper_1205_2933_gb300.inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("Ls,bound", [(12, 2.6e-6), (6, 2.6e-6), (24, 2.6e-6), (8, 6.8e-6)])
def test_basis_rounding(Ls, bound):
    from gpu_util import ctx_for
    from paper_1205_2933_gb300 import dwfmg as G
    dims, nvec = (4, 4, 8, 4), 16
    start = torch.from_numpy(I.random_vectors(nvec // 2, dims, Ls, 3)).cuda()
    q = []
    for prec in (G.DWF_F64, G.DWF_F32):
        ctx = ctx_for(I.epsilon_links(dims, 0.5, 1), dims, Ls, 1.8, 0.1)
        p = G.mg_default_params()
        p.setup_iters0, p.smoother_prec = 8, prec
        G.mg_setup(ctx.h, 2, [nvec], [(2, 2, 2, 2)], p, start)
        q.append(torch.empty(nvec * ctx.field_elems, dtype=torch.complex128, device="cuda"))
        G.mg_get_vectors(ctx.h, 0, q[-1])
        torch.cuda.synchronize()
        ctx.close()
    assert ((q[1] - q[0]).norm() / q[0].norm()).item() < bound
