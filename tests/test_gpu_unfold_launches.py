"""bgw_unfold_spinor forms the phases in a launch of their own in large calls and
inside the one launch of small ones: the same bits, on both sides of the switch
(152 blocks of 256 plane waves x 8 bands)."""
import numpy as np
import pytest

from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [400, 401, 408, 409, 700])         # 150, 153, 153, 156 and 264 blocks
def test_large_call_equals_small_calls(gpu_lib, nb):
    torch = pytest.importorskip("torch")
    avec = syn.make_problem("si18_qx").avec
    at = np.asarray(avec).T
    rot = np.rint(np.linalg.inv(at) @ np.array([[0, 0, 1], [1, 0, 0], [0, 1, 0]]) @ at).astype(np.int32)
    rng = np.random.default_rng(nb)
    ngw = 600
    g = rng.integers(-9, 10, (ngw, 3)).astype(np.int32)
    tau = np.array([0.21, 0.4, 0.125])
    c = torch.from_numpy(rng.standard_normal((nb, 2, ngw)) + 1j * rng.standard_normal((nb, 2, ngw))).cuda()
    whole, parts = torch.empty_like(c), torch.empty_like(c)
    gpu_lib.bgw_unfold_spinor(avec, rot, tau, g, c, whole)
    for n in range(0, nb, 50):
        gpu_lib.bgw_unfold_spinor(avec, rot, tau, g, c[n:n + 50], parts[n:n + 50])
    torch.cuda.synchronize()
    assert torch.equal(whole, parts)
