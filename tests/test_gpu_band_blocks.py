"""bgw_mtxel_spinor on blocks of bands whose pair count is not a multiple of
the context's valence count: the scratch of the z and y passes must hold
every pair of the block (it was sized from the pair count divided by the
context's valence bands, and could come out some pairs short)."""
import numpy as np
import pytest

import oracle
from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

TOL_M = {"fp64": 1e-12, "mixed": 5e-6}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("v0, nv, c0, nc", [(0, 4, 3, 13), (2, 5, 0, 7), (7, 1, 23, 1), (1, 7, 1, 23)])
def test_mtxel_block_matches_oracle(gpu_lib, prec, v0, nv, c0, nc):
    torch = pytest.importorskip("torch")
    p = syn.make_problem("si18_qx")
    q, geps, _ = p.qs[0]
    ik = 4
    kp, G0 = oracle.umklapp(p.kcrys, ik, q)
    ref = oracle.mtxel(p.box, p.gvec[ik], p.coeff[ik][v0:v0 + nv], p.gvec[kp],
                       p.coeff[kp][p.nv + c0:p.nv + c0 + nc], G0, geps)
    ctx = gpu_lib.Chi0Context(p, prec)
    ctx.upload()
    M = torch.zeros((nv, nc, len(geps)), dtype=torch.complex128 if prec == "fp64" else torch.complex64, device="cuda")
    gpu_lib.bgw_mtxel_spinor(ctx.ctx, q, geps, ik, v0, nv, c0, nc, M)
    ctx.close()
    assert np.abs(M.cpu().numpy() - ref).max() <= TOL_M[prec] * np.abs(ref).max()


def test_alternating_spheres(gpu_lib):
    """The sphere map is copied to the device only when it changes: the same
    sphere twice, another of the same size, then the first again."""
    torch = pytest.importorskip("torch")
    p = syn.make_problem("si18_qx", nv=2, nc=3)
    q, a, _ = p.qs[0]
    b = np.ascontiguousarray(a[::-1])                       # same vectors, another order
    ctx = gpu_lib.Chi0Context(p, "fp64")
    ctx.upload()

    def call(g):
        M = torch.zeros((2, 3, len(g)), dtype=torch.complex128, device="cuda")
        gpu_lib.bgw_mtxel_spinor(ctx.ctx, q, g, 0, 0, 2, 0, 3, M)
        return M

    first, again, other, back = call(a), call(a), call(b), call(a)
    torch.cuda.synchronize()
    ctx.close()
    assert torch.equal(first, again) and torch.equal(first, back)
    assert torch.equal(first, other.flip(2)) and not torch.equal(first, other)
