"""Matrix-element calls inside a captured graph: the copy of the sphere map reads
its host source at every replay, so the source must outlive the call.  Captured
calls on two spheres replay to the bits of the eager calls, after other spheres
went through the same buffer and host memory was reused."""
import numpy as np
import pytest

from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_captured_matrix_elements(gpu_lib, prec):
    torch = pytest.importorskip("torch")
    p = syn.make_problem("si18_qx", nv=3, nc=5)
    q, a, _ = p.qs[0]
    b = np.ascontiguousarray(a[::-1])
    s = torch.cuda.Stream()
    ctx = gpu_lib.Chi0Context(p, prec, s)
    ctx.upload()
    dt = torch.complex128 if prec == "fp64" else torch.complex64
    Ms = torch.zeros((2, 3, 5, len(a)), dtype=dt, device="cuda")
    Mb = torch.zeros((8, 8, len(a)), dtype=dt, device="cuda")
    torch.cuda.synchronize()

    def calls():
        gpu_lib.bgw_mtxel_spinor(ctx.ctx, q, a, 0, 0, 3, 0, 5, Ms[0])
        gpu_lib.bgw_mtxel_spinor(ctx.ctx, q, b, 0, 0, 3, 0, 5, Ms[1])
        gpu_lib.bgw_mtxel_bands(ctx.ctx, q, a, 0, 0, 8, 0, 8, Mb)

    calls()
    s.synchronize()
    eager = Ms.cpu(), Mb.cpu()
    gpu_lib.bgw_graph_begin(ctx.ctx)
    calls()
    gpu_lib.bgw_graph_end(ctx.ctx)
    for i in range(3):
        junk = [np.full(n, 7, np.int32) for n in range(1000, 9000, 50)]      # host memory of the calls, reused
        c = np.ascontiguousarray(np.roll(a, i + 1, axis=0))
        gpu_lib.bgw_mtxel_spinor(ctx.ctx, q, c, 0, 0, 3, 0, 5, Ms[0])
        s.synchronize()
        Ms.zero_()
        Mb.zero_()
        torch.cuda.synchronize()
        gpu_lib.bgw_graph_launch(ctx.ctx)
        s.synchronize()
        assert torch.equal(Ms.cpu(), eager[0]) and torch.equal(Mb.cpu(), eager[1])
        del junk
    gpu_lib.bgw_mtxel_spinor(ctx.ctx, q, b, 0, 0, 3, 0, 5, Ms[0])            # eager again
    s.synchronize()
    assert torch.equal(Ms[0].cpu(), eager[0][1])
    ctx.close()
