"""Digit products (bgw_dz.cu) where one operand grows along G as the other falls:
an interaction that is huge at G = 0 against matrix elements that nearly vanish
there (states orthogonal up to 2^-20, as at small q).  Digits are cut on a scale
per row, so the large entries of one operand must not cost the other's digits.
Compared with extended precision over the library's own matrix elements.

Tolerance, against the sum of the magnitudes of an element's terms: K^X has the
weight, the product and the result rounded once each, K^D two products more;
4 and 8 roundings of FP64."""
import numpy as np
import pytest

from paper_2206_00808_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

ORTH, HEAD = 2.0 ** -20, 2.0 ** 40


def setup(B, torch, nv, nc, ng):
    p = syn.make_problem("si18_qx", nv=nv, nc=nc)
    rng = np.random.default_rng(ng)
    for k in range(p.nk):
        shape = p.coeff[k].shape
        c = np.linalg.qr(np.asarray(p.coeff[k]).reshape(shape[0], -1).T)[0].T
        mix = rng.standard_normal((shape[0], shape[0])) + 1j * rng.standard_normal((shape[0], shape[0]))
        p.coeff[k] = np.ascontiguousarray((c + ORTH * mix @ c).reshape(shape))
    ctx = B.Chi0Context(p, "fp64")
    ctx.upload()
    g = syn.eps_sphere(syn.reciprocal(p.avec), np.zeros(3), ng)
    assert not np.any(g[0])

    def elements(ik, a0, na, b0, nb):
        M = torch.zeros((na, nv + nc, ng), dtype=torch.complex128, device="cuda")
        B.bgw_mtxel_bands(ctx.ctx, np.zeros(3), g, ik, a0, na, 0, nv + nc, M)
        return np.ascontiguousarray(M.cpu().numpy()[:, b0:b0 + nb]).reshape(na * nb, ng)

    return p, ctx, g, elements


def long_product(a, b):
    """a b^T in extended precision, complex as (re, im)."""
    ar, ai, br, bi = (np.asarray(x, np.longdouble) for x in (*a, *b))
    return ar @ br.T - ai @ bi.T, ar @ bi.T + ai @ br.T


def check(got, ref, bound, roundings):
    tol = roundings * 2.0 ** -53 * bound
    assert (np.abs(got.real - ref[0]) <= tol).all() and (np.abs(got.imag - ref[1]) <= tol).all()


@pytest.mark.parametrize("ng", [33, 137])
def test_exchange_with_a_large_head(gpu_lib, ng):
    torch = pytest.importorskip("torch")
    nv, nc = 3, 4
    p, ctx, g, elements = setup(gpu_lib, torch, nv, nc, ng)
    v = np.random.default_rng(1).uniform(0.5, 1.5, ng)
    v[0] = HEAD
    KX = torch.zeros((nv * nc, nv * nc), dtype=torch.complex128, device="cuda")
    gpu_lib.bgw_bse_kernel(ctx.ctx, 1, 2, np.zeros(3), g, v, np.zeros(3), g, None, 0, nv, 0, nc, KX, None)
    mi, mj = elements(1, 0, nv, nv, nc), elements(2, 0, nv, nv, nc)
    got = KX.cpu().numpy() * p.nk                     # nk = 8: exact
    ctx.close()
    assert p.nk == 8
    vl = v.astype(np.longdouble)
    ref = long_product((mi.real * vl, mi.imag * vl), (mj.real, -mj.imag))
    check(got, ref, (np.abs(mi) * v) @ np.abs(mj).T, 4)


@pytest.mark.parametrize("ng", [33, 137])
def test_direct_with_a_large_head(gpu_lib, ng):
    torch = pytest.importorskip("torch")
    nv, nc, ik = 3, 4, 1
    p, ctx, g, elements = setup(gpu_lib, torch, nv, nc, ng)
    rng = np.random.default_rng(2)
    s = np.ones(ng)
    s[0] = np.sqrt(HEAD)
    W = rng.standard_normal((ng, ng)) + 1j * rng.standard_normal((ng, ng))
    W = np.ascontiguousarray(0.5 * (W + W.conj().T) * s[:, None] * s[None, :])
    KD = torch.zeros((nv * nc, nv * nc), dtype=torch.complex128, device="cuda")
    gpu_lib.bgw_bse_kernel(ctx.ctx, ik, ik, np.zeros(3), g, s, np.zeros(3), g, torch.from_numpy(W).cuda(), 0, nv, 0, nc,
                           None, KD)
    cc, vv = elements(ik, nv, nc, nv, nc), elements(ik, 0, nv, 0, nv)
    got = -KD.cpu().numpy() * p.nk
    ctx.close()
    y = long_product((vv.real, vv.imag), (W.real, W.imag))           # Y[(v v')][G]
    t = long_product((cc.real, -cc.imag), y)                         # [(c c')][(v v')]
    bound = np.abs(cc) @ np.abs(W) @ np.abs(vv).T

    def to_block(x):                                                 # [(v c)][(v' c')]
        return np.asarray(x).reshape(nc, nc, nv, nv).transpose(2, 0, 3, 1).reshape(nv * nc, nv * nc)

    check(got, [to_block(x) for x in t], to_block(bound), 8)
