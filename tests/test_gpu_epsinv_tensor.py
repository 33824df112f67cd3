"""bgw_epsinv around the switch to tensor-core products (96 rows) and at sizes
that end in short blocks (32) and tiles (128 rows, 32 columns), against numpy's
LU in FP64.

Tolerance: eps~ = I + B B^H here has condition number below 50; an FP64 inverse
by either route is then off by at most about kappa n 2^-53 of its largest entry,
5e-13 at n = 300 in the worst case."""
import numpy as np
import pytest

from paper_2206_00808_gb300 import synthetic as syn  # noqa: F401  (the package must import)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ng, nf", [(95, 2), (96, 1), (97, 3), (128, 2), (129, 1), (193, 2), (300, 3)])
@pytest.mark.parametrize("mode", ["epsinv_sym", "W", "epsinv"])
def test_epsinv_matches_lu(gpu_lib, ng, nf, mode):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(ng)
    s = rng.uniform(0.2, 2.0, ng)
    chi = np.empty((nf, ng, ng), dtype=np.complex128)
    for j in range(nf):
        b = (rng.standard_normal((ng, ng)) + 1j * rng.standard_normal((ng, ng))) / np.sqrt(ng) / s[:, None]
        chi[j] = -(b @ b.conj().T) * 2.0 / (1 + j)
    dev = torch.from_numpy(chi).cuda()
    gpu_lib.bgw_epsinv(dev, s, mode)
    left, right = {"epsinv_sym": (1 + 0 * s, 1 + 0 * s), "W": (s, s), "epsinv": (s, 1 / s)}[mode]
    for j in range(nf):
        ref = left[:, None] * np.linalg.inv(np.eye(ng) - s[:, None] * chi[j] * s[None, :]) * right[None, :]
        assert np.abs(dev[j].cpu().numpy() - ref).max() <= 5e-13 * np.abs(ref).max()


def test_epsinv_rejects_an_indefinite_matrix(gpu_lib):
    torch = pytest.importorskip("torch")
    chi = torch.zeros((1, 130, 130), dtype=torch.complex128, device="cuda")
    chi[0].diagonal()[77] = 5.0                        # 1 - s chi s < 0
    with pytest.raises(gpu_lib.BgwError) as e:
        gpu_lib.bgw_epsinv(chi, np.ones(130))
    assert e.value.status == gpu_lib.BGW_E_ARG and "pivot" in str(e.value)
