"""A self-energy whose digit product is cut into pieces of both operands (more
than 512 MiB of digits each): 64 bands times 56 against 5000 G on an 18^3 box,
compared with the same sums in FP64 on the library's own matrix elements.

Tolerance: two nested sums of 5000 terms on the FP64 side, 2 5000 2^-53 of the
sum of the magnitudes."""
import numpy as np
import pytest

from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def test_sigma_in_pieces(gpu_lib):
    torch = pytest.importorskip("torch")
    B = gpu_lib
    ng, nv, nc, n0, nn = 5000, 8, 56, 4, 56
    p = syn.make_problem("si18_qx", nv=nv, nc=nc)
    q = np.asarray(p.qs[0][0])
    g = np.stack(np.meshgrid(*[np.arange(-9, 9)] * 3, indexing="ij"), -1).reshape(-1, 3).astype(np.int32)[:ng]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    W = torch.randn((ng, ng), dtype=torch.complex128, device="cuda", generator=gen)
    W = 0.5 * (W + W.mH)
    v = np.random.default_rng(5).uniform(0.1, 3.0, ng)
    ctx = B.Chi0Context(p, "fp64")
    ctx.upload()
    ik = 4
    sx, coh = B.bgw_sigma_cohsex(ctx.ctx, q, g, ik, n0, nn, W.contiguous(), v)
    jk = next(j for j in range(p.nk) if np.abs(np.mod(p.kcrys[j] + q - p.kcrys[ik] + 0.5, 1.0) - 0.5).max() < 1e-6)
    M = torch.zeros((nv + nc, nn, ng), dtype=torch.complex128, device="cuda")
    B.bgw_mtxel_bands(ctx.ctx, q, g, jk, 0, nv + nc, n0, nn, M)
    torch.cuda.synchronize()
    ctx.close()
    Y = (M.view(-1, ng) @ W.T).view_as(M)
    pair = (M.conj() * Y).sum(2).real
    size = M.abs().sum(2).max().item() ** 2 * W.abs().max().item()        # above every pair's sum of magnitudes
    bare = (M.abs().square() * torch.from_numpy(v).cuda()).sum(2)
    want_sx = -pair[:nv].sum(0).cpu().numpy() / p.nk
    want_coh = 0.5 * (pair.sum(0) - bare.sum(0)).cpu().numpy() / p.nk
    tol = 2 * ng * 2.0 ** -53 * size * (nv + nc) / p.nk
    assert tol < 1e-3 * np.abs(want_coh).max()
    assert np.abs(sx - want_sx).max() <= tol and np.abs(coh - want_coh).max() <= tol
