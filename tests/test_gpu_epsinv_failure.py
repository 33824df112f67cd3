"""bgw_epsinv whose first digit product loses an operand load (BGW_FAULT =
drop@epsinv): the bounded wait gives up, the call reports BGW_E_TIMEOUT within
seconds, and the next call is right."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_dropped_load_reports_timeout(gpu_lib, monkeypatch):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(2)
    ng = 150
    b = (rng.standard_normal((ng, ng)) + 1j * rng.standard_normal((ng, ng))) / np.sqrt(ng)
    chi, s = -(b @ b.conj().T)[None], rng.uniform(0.5, 2.0, ng)
    ref = np.linalg.inv(np.eye(ng) - s[:, None] * chi[0] * s[None, :])
    monkeypatch.setenv("BGW_FAULT", "drop@epsinv")
    t0 = time.time()
    with pytest.raises(gpu_lib.BgwError) as e:
        gpu_lib.bgw_epsinv(torch.from_numpy(chi).cuda(), s, "epsinv_sym")
    assert e.value.status == gpu_lib.BGW_E_TIMEOUT and time.time() - t0 < 60
    monkeypatch.delenv("BGW_FAULT")
    dev = torch.from_numpy(chi).cuda()
    gpu_lib.bgw_epsinv(dev, s, "epsinv_sym")
    assert np.abs(dev[0].cpu().numpy() - ref).max() <= 5e-13 * np.abs(ref).max()
