"""FP64 transforms in 64-bit fixed point (one scale per line, or per band and
x-plane): matrix elements against the CPU FP64 oracle on every box length and
on boxes whose planes are not square, with kept outputs inside and outside the
compile-time window, part-filled pair tiles, and bands of very different size.

Tolerance: a line's fixed-point error is below 2^-53 of its rms and each of
the six passes (three per transform) rounds its FP64 output once, so M is off
by a few 2^-53 of max |M|; the oracle's sum of a few thousand products adds as
much.  1e-14 of max |M| leaves a factor of ten over both."""
import numpy as np
import pytest

import oracle
from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

TOL = 1e-14


def mtxel(gpu_lib, torch, p, ik, v0, nv, c0, nc):
    q, geps, _ = p.qs[0]
    ctx = gpu_lib.Chi0Context(p, "fp64")
    ctx.upload()
    M = torch.zeros((nv, nc, len(geps)), dtype=torch.complex128, device="cuda")
    gpu_lib.bgw_mtxel_spinor(ctx.ctx, q, geps, ik, v0, nv, c0, nc, M)
    ctx.close()
    return M.cpu().numpy()


def reference(p, ik, v0, nv, c0, nc):
    q, geps, _ = p.qs[0]
    kp, G0 = oracle.umklapp(p.kcrys, ik, q)
    return oracle.mtxel(p.box, p.gvec[ik], p.coeff[ik][v0:v0 + nv], p.gvec[kp],
                        p.coeff[kp][p.nv + c0:p.nv + c0 + nc], G0, geps)


@pytest.mark.parametrize("box, ng, nv, nc", [
    ((16, 16, 16), 137, 3, 5), ((18, 18, 18), 137, 2, 4), ((20, 20, 20), 137, 1, 1), ((24, 24, 24), 137, 3, 9),
    ((27, 27, 27), 137, 2, 5), ((30, 30, 30), 137, 3, 7), ((32, 32, 32), 137, 5, 4), ((36, 36, 36), 137, 3, 3),
    ((40, 40, 40), 137, 1, 5),
    ((24, 24, 24), 1500, 2, 5), ((32, 32, 32), 1500, 3, 4),      # kept outputs beyond +-8
    ((16, 20, 20), 89, 2, 5), ((48, 24, 24), 89, 2, 5),          # square planes, another first axis
    ((20, 24, 18), 89, 3, 4), ((36, 27, 40), 89, 2, 3),          # no square planes: the single passes
])
def test_mtxel_matches_oracle(gpu_lib, box, ng, nv, nc):
    torch = pytest.importorskip("torch")
    p = syn.make_problem("si18_qx", box=box, ng=ng, nv=nv, nc=nc + 1, ecut_wfn=22.0)
    for ik in (0, 4):                                            # 4: the umklapp k
        got, ref = mtxel(gpu_lib, torch, p, ik, 0, nv, 1, nc), reference(p, ik, 0, nv, 1, nc)
        assert np.abs(got - ref).max() <= TOL * np.abs(ref).max()


def test_scales_and_non_finite_bands(gpu_lib):
    """A power of two in a band's coefficients comes out as that power, bit for
    bit; a zero band gives zeros; a NaN or infinite coefficient makes its band's
    elements NaN and leaves the others' bits alone."""
    torch = pytest.importorskip("torch")
    p = syn.make_problem("si18_qx", nv=4, nc=5)
    base = mtxel(gpu_lib, torch, p, 0, 0, 4, 0, 5)
    for c in p.coeff:
        c[1] *= 2.0 ** -250
        c[2] = 0.0
        c[p.nv + 3] *= 2.0 ** 200
        c[p.nv + 4][0, 7] = complex(np.nan, 1.0)
        c[0][1, 3] = complex(0.0, np.inf)
    got = mtxel(gpu_lib, torch, p, 0, 0, 4, 0, 5)
    scale = np.ones((4, 5))
    scale[1] = 2.0 ** -250
    scale[:, 3] *= 2.0 ** 200
    assert np.isnan(got[0]).all() and np.isnan(got[:, 4]).all()
    assert (got[2, :4] == 0).all()
    for v in (1, 3):
        assert (got[v, :4] == base[v, :4] * scale[v, :4, None]).all()


def test_small_spin_components_keep_their_precision(gpu_lib):
    """A nearly spin-up valence band against spin-down conduction bands: the
    element comes from the small components alone and is as exact as any."""
    torch = pytest.importorskip("torch")
    p = syn.make_problem("si18_qx", nv=3, nc=4)
    for c in p.coeff:
        c[:p.nv, 1] *= 2.0 ** -40                # valence: spin down 1e-12 of spin up
        c[p.nv:, 0] = 0.0                        # conduction: spin down only
        c[p.nv + 1, 0] = c[p.nv + 1, 1] * 2.0 ** -50
    got, ref = mtxel(gpu_lib, torch, p, 4, 0, 3, 0, 4), reference(p, 4, 0, 3, 0, 4)
    assert np.abs(got - ref).max() <= TOL * np.abs(ref).max()
