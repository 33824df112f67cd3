"""bgw_epsinv on badly scaled matrices (s_0 far above or below the others, as a
metal's head at small q; s falling over many orders): the inverse keeps its
accuracy entry by entry on the scales of eps~'s diagonal.

Tolerance: with B = X eps~ X of unit-size diagonal, an FP64 inverse by either
route is off by at most about kappa(B) n 2^-53 of the largest entry of B^-1."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ng", [96, 129, 200])
@pytest.mark.parametrize("head, fall", [(30, 0), (20, 0), (-30, 0), (0, 40), (-20, -60)])
@pytest.mark.parametrize("mode", ["epsinv_sym", "W", "epsinv"])
def test_badly_scaled_matrix(gpu_lib, ng, head, fall, mode):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(ng)
    s = rng.uniform(0.5, 2.0, ng) * 2.0 ** (-fall * np.arange(ng) / ng)
    s[0] = 2.0 ** head
    b = (rng.standard_normal((2, ng, ng)) + 1j * rng.standard_normal((2, ng, ng))) / np.sqrt(ng)
    chi = -(b @ b.conj().transpose(0, 2, 1))
    chi[1] *= 0.25
    dev = torch.from_numpy(chi).cuda()
    gpu_lib.bgw_epsinv(dev, s, mode)
    got = dev.cpu().numpy()
    left, right = {"epsinv_sym": (1 + 0 * s, 1 + 0 * s), "W": (s, s), "epsinv": (s, 1 / s)}[mode]
    for j in range(2):
        eps = np.eye(ng) - s[:, None] * chi[j] * s[None, :]
        x = 2.0 ** -np.rint(0.5 * np.log2(eps.diagonal().real))
        B = x[:, None] * eps * x[None, :]
        ref = np.linalg.inv(B)
        kappa = np.linalg.norm(B, 2) * np.linalg.norm(ref, 2)
        mine = got[j] / left[:, None] / right[None, :] / x[:, None] / x[None, :]
        assert np.abs(mine - ref).max() <= kappa * ng * 2.0 ** -53 * np.abs(ref).max()
