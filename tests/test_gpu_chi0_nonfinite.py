"""FP64 chi0 of states or energies with an infinity or a NaN: every pair of such a
band is not finite at any G, so the whole sum is NaN (the digits of the
tensor-core contraction must not turn it into numbers), as on the FP64 pipe;
good inputs afterwards give the good sum."""
import numpy as np
import pytest

import oracle
from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", ["valence", "conduction", "energy"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("form", [0, 1])
def test_bad_band_gives_nan(gpu_lib, where, bad, form):
    p = syn.make_problem("si18_qx", nv=3, nc=5, nfreq=2)
    ref = oracle.chi0(p)
    good = p.coeff[2], p.energy[2]
    c, e = np.array(good[0]), np.array(good[1])
    if where == "energy":
        e[1] = np.nan                       # (an infinite energy has weight 0)
    else:
        c[1 if where == "valence" else p.nv + 2, 1, 7] = bad
    p.coeff[2], p.energy[2] = c, e
    ctx = gpu_lib.Chi0Context(p, "fp64")
    gpu_lib.bgw_set_option(ctx.ctx, gpu_lib.BGW_OPT_FP64_CONTRACTION, form)
    gpu_lib.bgw_set_option(ctx.ctx, gpu_lib.BGW_OPT_KCHUNK, 3)
    ctx.upload()
    ctx.accumulate()
    assert np.isnan(ctx.finalize()).all()
    p.coeff[2], p.energy[2] = good
    ctx.upload(ks=[2])
    ctx.reset()
    ctx.accumulate()
    got = ctx.finalize()
    ctx.close()
    assert np.linalg.norm(got - ref) <= 1e-10 * np.linalg.norm(ref)
