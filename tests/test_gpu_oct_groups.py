"""Eight-lane z + y kernel (cubic 48 and 64 boxes) with one, two and four
conduction bands per CTA and a last group that is not full: a block of matrix
elements equals the same block taken one conduction band at a time, which always
runs one band per CTA.

Tolerance: the two forms do the same operations; a few roundings of the largest
element, should the compiler contract them differently."""
import numpy as np
import pytest

import oracle
from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

TOL = {"fp64": 4 * 2.0 ** -53, "mixed": 4 * 2.0 ** -24}


@pytest.mark.parametrize("box", [48, 64])
@pytest.mark.parametrize("prec, nv, nc", [("mixed", 1, 2), ("mixed", 1, 4), ("mixed", 1, 5), ("mixed", 3, 7), ("mixed", 2, 9),
                                          ("fp64", 1, 5), ("fp64", 3, 7), ("fp64", 8, 41)])
def test_block_equals_single_bands(gpu_lib, box, prec, nv, nc):
    torch = pytest.importorskip("torch")
    p = syn.make_problem("si18_qx", box=(box,) * 3, nv=nv, nc=nc)
    q, geps, _ = p.qs[0]
    ik = 4
    kp, _ = oracle.umklapp(p.kcrys, ik, q)
    ctx = gpu_lib.Chi0Context(p, prec)
    ctx.upload(ks=sorted({ik, kp}))
    dt = torch.complex128 if prec == "fp64" else torch.complex64
    M = torch.zeros((nv, nc, len(geps)), dtype=dt, device="cuda")
    gpu_lib.bgw_mtxel_spinor(ctx.ctx, q, geps, ik, 0, nv, 0, nc, M)
    scale = M.abs().max().item()
    assert scale > 0
    for c in range(nc):
        one = torch.zeros((nv, 1, len(geps)), dtype=dt, device="cuda")
        gpu_lib.bgw_mtxel_spinor(ctx.ctx, q, geps, ik, 0, nv, c, 1, one)
        assert (one[:, 0] - M[:, c]).abs().max().item() <= TOL[prec] * scale
    ctx.close()
