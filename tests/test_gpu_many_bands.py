"""FP64 contexts with integer grids and more bands than a launch has blocks along
y and z (65535): bands that are one plane wave each, so that every matrix element
is conj(c_v) c_c at G = 0 and 0 elsewhere.  131075 valence bands are more than
65535 tiles of two."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k1_path", [0, 1])
def test_more_bands_than_grid_blocks(gpu_lib, k1_path):
    torch = pytest.importorskip("torch")
    B = gpu_lib
    nv, nc = 131075, 2
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 40 GB on the device")
    i = np.arange(nv + nc)
    c = np.zeros((nv + nc, 2, 1), np.complex128)
    c[:, 0, 0] = 1.0 + 1e-3 * (i % 997) + 0.5j
    c[:, 1, 0] = 0.25j * (1 + i % 3)
    ctx = B.bgw_create((16, 16, 16), np.zeros((1, 3)), nv, nc, "fp64")
    B.bgw_set_option(ctx, B.BGW_OPT_K1_PATH, k1_path)
    B.bgw_wfn_upload(ctx, 0, np.zeros((1, 3), np.int32), torch.from_numpy(c).cuda(),
                     torch.from_numpy(np.where(i < nv, -1.0, 1.0)).cuda())
    M = torch.zeros((nv, nc, 2), dtype=torch.complex128, device="cuda")
    B.bgw_mtxel_spinor(ctx, np.zeros(3), np.array([[0, 0, 0], [1, 0, 0]], np.int32), 0, 0, nv, 0, nc, M)
    got = M.cpu().numpy()
    B.bgw_destroy(ctx)
    ref = np.einsum("vs,cs->vc", c[:nv, :, 0].conj(), c[nv:, :, 0])
    assert np.abs(got[..., 0] - ref).max() <= 1e-14 * np.abs(ref).max()
    assert np.abs(got[..., 1]).max() <= 1e-14 * np.abs(ref).max()
