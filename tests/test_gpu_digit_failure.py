"""A digit product (bgw_dz.cu) whose bounded device wait runs out: the calls that
use it report it, or leave NaN, and the error word of the chi0 sum is left alone
in both directions.  The wait runs out because block 0 skips its first operand
loads (BGW_OPT_TEST_DROP_LOAD = 1 in an FP64 context)."""
import numpy as np
import pytest

import oracle
from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

IK, N0, NN = 4, 2, 3


def hermitian(n):
    rng = np.random.default_rng(n)
    a = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    return np.ascontiguousarray(0.5 * (a + a.conj().T))


def setup(gpu_lib, torch):
    p = syn.make_problem("si18_qx", nv=4, nc=8)
    ctx = gpu_lib.Chi0Context(p, "fp64")
    ctx.upload()
    return p, ctx, torch.from_numpy(hermitian(len(p.qs[0][1]))).cuda()


def test_sigma_reports_its_own_wait_and_keeps_the_error_of_chi0(gpu_lib):
    torch = pytest.importorskip("torch")
    p, ctx, W = setup(gpu_lib, torch)
    q, geps, _ = p.qs[0]
    v = np.full(len(geps), 0.5)
    good = gpu_lib.bgw_sigma_cohsex(ctx.ctx, q, geps, IK, N0, NN, W, v)
    p.energy[0] = np.array(p.energy[0])
    p.energy[0][0] = 90.0                               # an occupied band above the empty ones
    ctx.upload(ks=[0])
    ctx.accumulate()                                    # records a positive pair weight
    gpu_lib.bgw_set_option(ctx.ctx, gpu_lib.BGW_OPT_TEST_DROP_LOAD, 1)
    sx, coh = np.full(NN, 7.0), np.full(NN, 8.0)
    with pytest.raises(gpu_lib.BgwError) as e:
        gpu_lib.bgw_sigma_cohsex(ctx.ctx, q, geps, IK, N0, NN, W, v, sx, coh)
    assert e.value.status == gpu_lib.BGW_E_TIMEOUT
    assert (sx == 7.0).all() and (coh == 8.0).all()
    gpu_lib.bgw_set_option(ctx.ctx, gpu_lib.BGW_OPT_TEST_DROP_LOAD, 0)
    again = gpu_lib.bgw_sigma_cohsex(ctx.ctx, q, geps, IK, N0, NN, W, v)
    assert np.array_equal(again[0], good[0]) and np.array_equal(again[1], good[1])
    with pytest.raises(gpu_lib.BgwError) as e:
        ctx.finalize()
    assert e.value.status == gpu_lib.BGW_E_ARG and "pair weight" in str(e.value)
    ctx.close()


def test_bse_reports_or_marks_its_own_wait_and_leaves_chi0_alone(gpu_lib):
    torch = pytest.importorskip("torch")
    p, ctx, W = setup(gpu_lib, torch)
    q, geps, _ = p.qs[0]
    z, v = np.zeros(3), np.full(len(geps), 0.5)
    n = p.nv * 8
    KX, KD = (torch.zeros((n, n), dtype=torch.complex128, device="cuda") for _ in range(2))

    def bse(kx, kd):
        gpu_lib.bgw_bse_kernel(ctx.ctx, IK, oracle.umklapp(p.kcrys, IK, q)[0], z, geps, v, q, geps, W, 0, p.nv, 0, 8, kx, kd)

    bse(KX, KD)
    good = KX.cpu(), KD.cpu()
    ctx.accumulate()
    gpu_lib.bgw_set_option(ctx.ctx, gpu_lib.BGW_OPT_TEST_DROP_LOAD, 1)
    with pytest.raises(gpu_lib.BgwError) as e:
        bse(KX, KD)
    assert e.value.status == gpu_lib.BGW_E_TIMEOUT
    assert torch.equal(KD.cpu(), good[1])               # not formed
    KD.zero_()
    torch.cuda.synchronize()
    bse(None, KD)
    assert torch.isnan(torch.view_as_real(KD)).any()
    gpu_lib.bgw_set_option(ctx.ctx, gpu_lib.BGW_OPT_TEST_DROP_LOAD, 0)
    got, ref = ctx.finalize(), oracle.chi0(p)
    assert np.linalg.norm(got - ref) <= 1e-10 * np.linalg.norm(ref)
    bse(KX, KD)
    assert torch.equal(KX.cpu(), good[0]) and torch.equal(KD.cpu(), good[1])
    ctx.close()
