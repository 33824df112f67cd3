"""FP64 complex products from BF16 digit slices (bgw_dz.cu), through the calls
that use them: the self-energy and the BSE kernel blocks against the CPU FP64
oracle, at sphere sizes around the switch from the FP64 kernel (32), the k'
blocks (16 complex) and the promotion of the sums (80 complex), and at row and
column counts around the 128-row and 32-column tiles.

Tolerance: a product's digits keep 2^-62 of its rows' scales and the result is
rounded once, so the matrix elements dominate: off by a few 2^-53 of max |M| in
both, which two or three factors and some hundred terms turn into a few 1e-15 of
the largest entry.  1e-13 leaves a factor of ten or more."""
import numpy as np
import pytest

import oracle
from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

TOL = 1e-13


def hermitian(rng, n):
    a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    s = np.exp(-4.0 * np.arange(n) / n)            # falls with G as an interaction does
    return 0.5 * (a + a.conj().T) * s[:, None] * s[None, :]


@pytest.mark.parametrize("ng, nv, nc", [(31, 3, 4), (32, 3, 4), (33, 5, 7), (80, 4, 8), (81, 8, 16), (137, 8, 17)])
def test_bse_kernel(gpu_lib, ng, nv, nc):
    torch = pytest.importorskip("torch")
    p = syn.make_problem("si18_qx", nv=nv, nc=nc)
    bvec = syn.reciprocal(p.avec)
    z, qd, ik, jk = np.zeros(3), np.array([0.5, 0, 0]), 4, 0        # an umklapp block
    geps0, gepsd = syn.eps_sphere(bvec, z, ng), syn.eps_sphere(bvec, qd, ng)
    v0 = oracle.coulomb(p.avec, z, geps0)
    W = hermitian(np.random.default_rng(ng), ng)
    KXr, KDr = oracle.bse_kernel(p, ik, jk, geps0, v0, qd, gepsd, W, (0, nv), (0, nc))
    ctx = gpu_lib.Chi0Context(p, "fp64")
    ctx.upload()
    KX = torch.zeros((nv * nc, nv * nc), dtype=torch.complex128, device="cuda")
    KD = torch.zeros_like(KX)
    gpu_lib.bgw_bse_kernel(ctx.ctx, ik, jk, z, geps0, v0, qd, gepsd, torch.from_numpy(np.ascontiguousarray(W)).cuda(),
                           0, nv, 0, nc, KX, KD)
    ctx.close()
    assert np.abs(KX.cpu().numpy() - KXr).max() <= TOL * np.abs(KXr).max()
    assert np.abs(KD.cpu().numpy() - KDr).max() <= TOL * np.abs(KDr).max()


@pytest.mark.parametrize("ng", [32, 81, 161])
def test_sigma_cohsex(gpu_lib, ng):
    torch = pytest.importorskip("torch")
    p = syn.make_problem("si18_qx", nv=5, nc=12, ng=ng)
    q, geps, _ = p.qs[0]
    rng = np.random.default_rng(ng)
    W, v = hermitian(rng, ng), rng.uniform(0.1, 3.0, ng)
    sx_ref, coh_ref = oracle.sigma_cohsex(p, 4, q, geps, W, v, 2, 9)
    ctx = gpu_lib.Chi0Context(p, "fp64")
    ctx.upload()
    sx, coh = gpu_lib.bgw_sigma_cohsex(ctx.ctx, q, geps, 4, 2, 9, torch.from_numpy(np.ascontiguousarray(W)).cuda(), v)
    ctx.close()
    scale = max(np.abs(sx_ref).max(), np.abs(coh_ref).max())
    assert np.abs(sx - sx_ref).max() <= TOL * scale
    assert np.abs(coh - coh_ref).max() <= TOL * scale
