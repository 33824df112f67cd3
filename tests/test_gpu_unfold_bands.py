"""bgw_unfold_spinor takes up to 65535 x 16 bands in one call (and refuses more):
the identity without a translation leaves spinors of two plane waves as they are."""
import numpy as np
import pytest

from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [7, 8, 65535 * 8 + 1, 65535 * 16])
def test_number_of_bands(gpu_lib, nb):
    torch = pytest.importorskip("torch")
    avec = syn.make_problem("si18_qx").avec
    g = np.array([[0, 0, 0], [1, -2, 3]], np.int32)
    c = torch.zeros((nb, 2, 2), dtype=torch.complex128, device="cuda")
    c.real.copy_(torch.arange(4 * nb, device="cuda", dtype=torch.float64).view(nb, 2, 2) % 65521 + 1.0)
    out = torch.zeros_like(c)
    gout = gpu_lib.bgw_unfold_spinor(avec, np.eye(3, dtype=np.int32), np.zeros(3), g, c, out)
    assert np.array_equal(gout, g)
    assert (out - c).abs().max().item() <= 4 * 2.0 ** -53 * 65521


def test_too_many_bands_are_refused(gpu_lib):
    torch = pytest.importorskip("torch")
    avec = syn.make_problem("si18_qx").avec
    c = torch.zeros((65535 * 16 + 1, 2, 1), dtype=torch.complex128, device="cuda")
    with pytest.raises(gpu_lib.BgwError) as e:
        gpu_lib.bgw_unfold_spinor(avec, np.eye(3, dtype=np.int32), np.zeros(3), np.zeros((1, 3), np.int32), c,
                                  torch.empty_like(c))
    assert e.value.status == gpu_lib.BGW_E_ARG
