"""Deferred builds of FP64 integer grids (BGW_OPT_DEFER_K1), several k-points per
launch: bitwise the eager grids for more k-points than one launch takes, for
k-points whose scratch needs more than one group, for k-points with spheres of
different sizes and for a box that is not a cube."""
import numpy as np
import pytest

from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(kgrid=(5, 5, 3), q=(0.2, 0, 0), nv=2, nc=3, ecut_wfn=12.0, ng=27),          # 75 k-points: 64 + 11
    dict(box=(32, 32, 32), nv=8, nc=122, ng=59),                                     # 130 bands: groups of a few
    dict(box=(40, 18, 18), nv=3, nc=4, ng=27),
], ids=["75k", "130bands", "40x18x18"])
def test_deferred_equals_eager(gpu_lib, kw):
    torch = pytest.importorskip("torch")
    B = gpu_lib
    p = syn.make_problem("si18_qx", **kw)
    p.gvec[1], p.coeff[1] = p.gvec[1][:20], np.ascontiguousarray(p.coeff[1][:, :, :20])     # a small sphere
    q, geps, nc = p.qs[0]
    got = {}
    for defer in (0, 1):
        ctx = B.Chi0Context(p, "fp64")
        B.bgw_set_option(ctx.ctx, B.BGW_OPT_DEFER_K1, defer)
        B.bgw_profile(ctx.ctx, True)
        ctx.upload()
        out = []
        for ik in range(p.nk):
            M = torch.zeros((p.nv, nc, len(geps)), dtype=torch.complex128, device="cuda")
            B.bgw_mtxel_spinor(ctx.ctx, q, geps, ik, 0, p.nv, 0, nc, M)
            out.append(M.cpu())
        calls = B.bgw_profile_read(ctx.ctx)["wfn_to_grid"][1]
        ctx.close()
        assert calls == p.nk if defer == 0 else calls < p.nk            # built together
        got[defer] = out
    for a, b in zip(got[0], got[1]):
        assert torch.equal(a, b)
