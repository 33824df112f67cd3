"""Digit products (bgw_dz.cu) over long sums whose terms all agree in sign and
digits: the exchange kernel of states that are one point in real space, whose
matrix elements are the same for every G (1/3 in both components for one pair),
up to the longest sum the digits take (5000) and the first that the FP64 kernel
takes (5001).  Compared with the sum in extended precision over the library's own
matrix elements.

Tolerance: the digits drop 2^-58 of the products' scale and the result is rounded
once, so 4 roundings of FP64 (4.5e-16); the FP64 kernel rounds each of n terms,
n 2^-53 of the sum of magnitudes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 18


@pytest.mark.parametrize("ng", [700, 1400, 4999, 5000, 5001])
def test_exchange_of_point_states(gpu_lib, ng):
    torch = pytest.importorskip("torch")
    B = gpu_lib
    g = np.stack(np.meshgrid(*[np.arange(-N // 2, N // 2)] * 3, indexing="ij"), -1).reshape(-1, 3).astype(np.int32)
    nv, nc = 2, 3
    factor = np.array([1.0, 0.7 - 0.2j, (1 + 1j) / 3, 0.4 + 0.9j, -0.6 + 0.1j]) / np.sqrt(N ** 3)
    coeff = np.broadcast_to(factor[:, None, None], (nv + nc, 2, len(g))) * np.sqrt(0.5)
    ctx = B.bgw_create((N, N, N), np.zeros((1, 3)), nv, nc, "fp64")
    B.bgw_wfn_upload(ctx, 0, g, np.ascontiguousarray(coeff), np.array([-2.0, -1.0, 1.0, 2.0, 3.0]))
    gs = np.ascontiguousarray(g[np.argsort((g.astype(np.int64) ** 2).sum(1), kind="stable")[:ng]])
    z, v = np.zeros(3), np.ones(ng)
    M = torch.zeros((nv, nc, ng), dtype=torch.complex128, device="cuda")
    KX = torch.zeros((nv * nc, nv * nc), dtype=torch.complex128, device="cuda")
    B.bgw_mtxel_spinor(ctx, z, gs, 0, 0, nv, 0, nc, M)
    B.bgw_bse_kernel(ctx, 0, 0, z, gs, v, z, gs, None, 0, nv, 0, nc, KX, None)
    m, got = M.cpu().numpy().reshape(nv * nc, ng), KX.cpu().numpy()
    B.bgw_destroy(ctx)
    assert np.allclose(m[0], (1 + 1j) / 3, rtol=1e-14, atol=0)
    re, im = m.real.astype(np.longdouble), m.imag.astype(np.longdouble)
    ref_re, ref_im = re @ re.T + im @ im.T, im @ re.T - re @ im.T
    scale = (np.abs(m) ** 2).sum(1)
    scale = np.sqrt(scale[:, None] * scale[None, :])
    tol = (4 if ng <= 5000 else ng) * 2.0 ** -53 * scale
    assert (np.abs(got.real - ref_re) <= tol).all() and (np.abs(got.imag - ref_im) <= tol).all()
