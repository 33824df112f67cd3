"""Digit products inside a captured graph: the direct BSE kernel (its products
leave their column exponents clear for the next one) replays to the bits of the
eager call, between eager calls on other operands."""
import numpy as np
import pytest

import oracle
from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def test_captured_direct_kernel(gpu_lib):
    torch = pytest.importorskip("torch")
    nv, nc, ik = 3, 7, 4
    p = syn.make_problem("si18_qx", nv=nv, nc=nc)
    q, g, _ = p.qs[0]
    ng = len(g)
    jk = oracle.umklapp(p.kcrys, ik, q)[0]
    rng = np.random.default_rng(4)
    s = 2.0 ** rng.integers(-12, 13, ng)                # graded, so that the columns matter
    W = rng.standard_normal((2, ng, ng)) + 1j * rng.standard_normal((2, ng, ng))
    W[0] *= s[:, None] * s[None, :]
    W = torch.from_numpy(W).cuda()
    v = np.ones(ng)
    st = torch.cuda.Stream()
    ctx = gpu_lib.Chi0Context(p, "fp64", st)
    ctx.upload()
    KD = torch.zeros((3, nv * nc, nv * nc), dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()

    def call(w, out):
        gpu_lib.bgw_bse_kernel(ctx.ctx, ik, jk, q, g, v, q, g, W[w], 0, nv, 0, nc, None, KD[out])

    call(0, 0)
    call(1, 1)
    st.synchronize()
    eager = KD.cpu()
    gpu_lib.bgw_graph_begin(ctx.ctx)
    call(0, 2)
    gpu_lib.bgw_graph_end(ctx.ctx)
    for _ in range(2):
        gpu_lib.bgw_graph_launch(ctx.ctx)
        st.synchronize()
        assert torch.equal(KD[2].cpu(), eager[0])
        KD[1:].zero_()
        torch.cuda.synchronize()
        call(1, 1)
        st.synchronize()
        assert torch.equal(KD[1].cpu(), eager[1])
    ctx.close()
