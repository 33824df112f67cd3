"""bgw_unfold_spinor where the two spin components of a plane wave have scales far
apart: each output keeps FP64 accuracy against the terms that it sums,
sum_k |U_rk| |c_k|, also where U is diagonal (a rotation about z), where the
smaller component is an output of its own.

Tolerance: four products and their sum in FP64, the phase (2 pi 2^-53) and its
product with U: below 16 roundings, 16 2^-53 of that sum."""
import numpy as np
import pytest

from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

Z4 = [[0, -1, 0], [1, 0, 0], [0, 0, 1]]
X2 = [[1, 0, 0], [0, -1, 0], [0, 0, -1]]
XYZ3 = [[0, 0, 1], [1, 0, 0], [0, 1, 0]]


@pytest.mark.parametrize("rot", [Z4, X2, XYZ3], ids=["z4", "x2", "xyz3"])
@pytest.mark.parametrize("ratio", [0, -8, -40, -300, 40])
def test_components_keep_their_own_accuracy(gpu_lib, rot, ratio):
    torch = pytest.importorskip("torch")
    avec = syn.make_problem("si18_qx").avec
    at = np.asarray(avec).T
    rot_lat = np.rint(np.linalg.inv(at) @ np.array(rot) @ at).astype(np.int32)
    rng = np.random.default_rng(3)
    nb, ngw = 11, 300
    g = rng.integers(-6, 7, (ngw, 3)).astype(np.int32)
    c = rng.standard_normal((nb, 2, ngw)) + 1j * rng.standard_normal((nb, 2, ngw))
    c[:, 1] *= 2.0 ** ratio
    c[3, 1, 5] = c[4, 0, 6] = 0.0                       # a component that is zero
    tau = np.array([0.25, 0.5, 0.125])
    cin = torch.from_numpy(c).cuda()
    out = torch.empty_like(cin)
    gout = gpu_lib.bgw_unfold_spinor(avec, rot_lat, tau, g, cin, out)
    U = np.asarray(gpu_lib.bgw_symmetry_su2(avec, rot_lat)[0]).reshape(-1).view(np.complex128).reshape(2, 2)
    phase = np.exp(-2j * np.pi * np.mod(gout @ tau, 1.0))
    ref = np.einsum("ab,nbg->nag", U, c) * phase
    bound = np.einsum("ab,nbg->nag", np.abs(U), np.abs(c))
    assert (np.abs(out.cpu().numpy() - ref) <= 16 * 2.0 ** -53 * bound).all()
