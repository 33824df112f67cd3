"""The calls a user of this library makes, at the sizes they make them.

A program that computes a GW self-energy or a Bethe-Salpeter spectrum with
this library uploads the spinor states of its k-points, sums chi0 over them
for one or several q, inverts the dielectric matrix, and takes matrix
elements, self-energies and BSE kernel blocks from the same states; before
that it may unfold states from the irreducible wedge.  The cases below are
those calls, from the smallest (one block of matrix elements on an 18^3 box)
to whole chi0 sums of the repository's own workloads (Si-like 24^3, GaSb-like
32^3, Bi2Se3-like 64^3), in both the FP64 and the mixed forms.

States are seeded complex Gaussians under a smooth kinetic-energy envelope,
each band normalised over both spinor components; energies are valence
U[-12, 0] and conduction U[1.1, 30] eV, sorted; frequencies linspace(0, 40)
eV on the imaginary axis.
"""
import functools
import math

import numpy as np
import torch

from paper_2206_00808_gb300 import binding as B

BOHR_PER_ANGSTROM = 1.0 / 0.529177210903
E2 = 27.211386245988          # e^2 in eV bohr
LENGTHS = (16, 18, 20, 24, 27, 30, 32, 36, 40, 48, 64)


# ------------------------------------------------------------------ geometry --

def _cell(case):
    if case["cell"] == "rhombohedral":          # Bi2Se3-like, hexagonal a and c
        a, c = 4.143 * BOHR_PER_ANGSTROM, 28.636 * BOHR_PER_ANGSTROM
        r = a / math.sqrt(3.0)
        return np.array([[a / 2, -r / 2, c / 3], [0.0, r, c / 3], [-a / 2, -r / 2, c / 3]])
    return 0.5 * case["a"] * np.array([[0.0, 1.0, 1.0], [1.0, 0.0, 1.0], [1.0, 1.0, 0.0]])


@functools.lru_cache(maxsize=None)
def _miller(key, k, radius2):
    """Miller triples with |k + h|^2 < radius2 and those squares, lexicographic."""
    avec = np.array(key).reshape(3, 3)
    bvec = 2.0 * np.pi * np.linalg.inv(avec).T
    r = [int(math.ceil(math.sqrt(radius2) * np.linalg.norm(avec[i]) / (2.0 * np.pi) + abs(k[i]))) + 1 for i in range(3)]
    g = np.stack(np.meshgrid(*[np.arange(-n, n + 1) for n in r], indexing="ij"), -1).reshape(-1, 3)
    e = (((np.array(k)[None, :] + g) @ bvec) ** 2).sum(1)
    keep = e < radius2
    return np.ascontiguousarray(g[keep].astype(np.int32)), e[keep]


def _sphere(case, k, ecut):
    return _miller(tuple(_cell(case).reshape(-1)), tuple(float(x) for x in k), float(ecut))


def _eps_sphere(case, q, ng):
    """The ng Miller vectors with the smallest |q + h|^2 (ties by order)."""
    radius2 = 1.0
    while True:
        g, e = _sphere(case, q, radius2)
        if len(g) >= ng:
            break
        radius2 *= 1.5
    order = np.lexsort((g[:, 2], g[:, 1], g[:, 0], np.round(e, 10)))
    return np.ascontiguousarray(g[order[:ng]])


def _kpoints(case):
    n = case["k1"], case["k2"], case["k3"]
    return np.array([(i / n[0], j / n[1], l / n[2]) for i in range(n[0]) for j in range(n[1]) for l in range(n[2])])


def _on_grid(case, k):
    """(index of the grid point k', G0) with k = k' + G0."""
    n = np.array([case["k1"], case["k2"], case["k3"]])
    m = np.rint(np.asarray(k) * n).astype(int)
    w = np.mod(m, n)
    return int((w[0] * n[1] + w[1]) * n[2] + w[2]), (m - w) // n


def _box(case):
    return case["n1"], case["n2"], case["n3"]


def _coulomb(case, q, gvec):
    """v(q + G) in eV, 0 where q + G = 0."""
    avec = _cell(case)
    bvec = 2.0 * np.pi * np.linalg.inv(avec).T
    g2 = (((np.asarray(q)[None, :] + gvec) @ bvec) ** 2).sum(1)
    return np.where(g2 > 1e-14, 4.0 * np.pi * E2 / abs(np.linalg.det(avec)) / np.where(g2 > 1e-14, g2, 1.0), 0.0)


# -------------------------------------------------------------------- inputs --

def _generator(seed, *more):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(np.random.SeedSequence([int(seed), *more]).generate_state(1)[0]))
    return g


def _randn(gen, *shape):
    return torch.randn(shape, dtype=torch.complex128, generator=gen, device="cuda")


def _states(case, seed, nb):
    """Per k: Miller list, coefficients [nb][2][ngw] and energies, on the device."""
    out = []
    for ik, k in enumerate(_kpoints(case)):
        g, e = _sphere(case, k, case["ecut"])
        z = _randn(_generator(seed, ik, 0), nb, 2, len(g))
        z *= torch.from_numpy(1.0 / (1.0 + (3.0 * e / case["ecut"]) ** 2)).cuda()
        z /= z.abs().square().sum((1, 2), keepdim=True).sqrt()
        rng = np.random.default_rng([int(seed), ik, 1])
        en = np.concatenate([np.sort(rng.uniform(-12.0, 0.0, case["nv"])), np.sort(rng.uniform(1.1, 30.0, nb - case["nv"]))])
        out.append((g, z, torch.from_numpy(en).cuda()))
    return out


def _frequencies(case):
    return np.linspace(0.0, 40.0, case["nfreq"]) if case["nfreq"] > 1 else np.zeros(1)


def _qlist(case):
    """[(q, dielectric sphere, conduction bands)]; several q differ in all three."""
    n = case["k1"], case["k2"], case["k3"]
    qs = []
    for i in range(case["nq"]):
        q = np.array([(case["q1"] + i) % n[0] / n[0], case["q2"] / n[1], (case["q3"] + (i + 1) // 2) % n[2] / n[2]])
        qs.append((q, _eps_sphere(case, q, case["ng"] - (31 * i) % max(1, case["ng"] // 4)), case["nc"] - (17 * i) % max(1, case["nc"] // 3)))
    return qs


def _screened(case, seed, q, gvec):
    """A static W = S eps~^-1 S (eV) and v(q + G): eps~ positive definite, its
    deviation from 1 falling with G as a dielectric matrix's does."""
    v = _coulomb(case, q, gvec)
    n = len(gvec)
    x = _randn(_generator(seed, 7, n), n, n + 8) / math.sqrt(n)
    x *= (4.0 / (1.0 + torch.arange(n, device="cuda", dtype=torch.float64) / 8.0)).sqrt()[:, None]
    w = torch.linalg.inv(torch.eye(n, dtype=torch.complex128, device="cuda") + x @ x.mH)
    s = torch.from_numpy(np.sqrt(v)).cuda()
    w = s[:, None] * (0.5 * (w + w.mH)) * s[None, :]
    return w.contiguous(), v


def _polarizability(case, seed):
    """chi0 of nfreq frequencies, Hermitian negative semidefinite, and sqrt(v)."""
    q = np.array([0.25, 0.0, 0.0])
    g = _eps_sphere(case, q, case["ng"])
    s = np.sqrt(_coulomb(case, q, g))
    n = case["ng"]
    damp = torch.from_numpy(1.0 / s).cuda() * (6.0 / (1.0 + torch.arange(n, device="cuda", dtype=torch.float64) / 16.0)).sqrt()
    chi = torch.empty((case["nfreq"], n, n), dtype=torch.complex128, device="cuda")
    x = _randn(_generator(seed, 3, n), n, n + 16) / math.sqrt(n)
    x *= damp[:, None]
    base = -(x @ x.mH)
    base = 0.5 * (base + base.mH)
    for j, w in enumerate(_frequencies(case)):
        chi[j] = base / (1.0 + (w / 12.0) ** 2)
    return chi, s


def _rotation(case):
    """A lattice symmetry of the FCC cell that is no inversion and turns by less
    than pi: three-fold about (1,1,1) or four-fold about z; and tau."""
    r = np.array([[0, 0, 1], [1, 0, 0], [0, 1, 0]]) if case["fold"] == 3 else np.array([[0, -1, 0], [1, 0, 0], [0, 0, 1]])
    at = _cell(case).T
    return r, np.rint(np.linalg.inv(at) @ r @ at).astype(np.int32), np.array([0.25, 0.25, 0.25])


# --------------------------------------------------------------------- cases --

def _si(**over):
    return dict(cell="fcc", a=10.26, k1=2, k2=2, k3=2, q1=1, q2=0, q3=0, nq=1, kchunk=1, **over)


def listed():
    return [
        # one small block of matrix elements: latency, launches and the host path
        _si(name="mtxel_si18_mixed_small", do="mtxel", prec="mixed", n1=18, n2=18, n3=18, ecut=28.1, nv=8, nc=24, nfreq=1,
            ng=137, ik=4, v0=0, v=8, c0=3, c=13),
        # a whole small chi0, as a convergence test runs it many times
        _si(name="chi0_si16_fp64", do="chi0", prec="fp64", n1=16, n2=16, n3=16, ecut=28.1, nv=8, nc=24, ng=137, nfreq=1),
        # the Si-like workload in both precisions: one q-point of a 4 x 4 x 4 grid
        dict(_si(name="chi0_si24_fp64", do="chi0", prec="fp64", n1=24, n2=24, n3=24, ecut=58.0, nv=8, nc=200, ng=350, nfreq=5),
             k1=4, k2=4, k3=4),
        dict(_si(name="chi0_si24_mixed", do="chi0", prec="mixed", n1=24, n2=24, n3=24, ecut=58.0, nv=8, nc=200, ng=350, nfreq=5),
             k1=4, k2=4, k3=4, kchunk=8),
        # the GaSb-like workload (all bands, G-vectors and frequencies) on 8 k-points
        dict(_si(name="chi0_gasb32_mixed", do="chi0", prec="mixed", n1=32, n2=32, n3=32, ecut=85.0, nv=18, nc=400, ng=800, nfreq=16),
             a=11.53, kchunk=2),
        # several ragged q-points in one call, as a screening run batches them
        dict(_si(name="chi0_batch32_mixed", do="chi0", prec="mixed", n1=32, n2=32, n3=32, ecut=85.0, nv=18, nc=341, ng=811, nfreq=5),
             a=11.53, k1=4, k2=1, k3=1, nq=3, kchunk=2),
        # a long rhombohedral cell on a 64^3 box with a large dielectric sphere
        dict(_si(name="chi0_bi2se3_64_mixed", do="chi0", prec="mixed", n1=64, n2=64, n3=64, ecut=67.9, nv=8, nc=125, ng=2000, nfreq=8),
             cell="rhombohedral", k2=1, k3=1),
        # a block of FP64 matrix elements of the GaSb-like states at an umklapp k
        dict(_si(name="mtxel_gasb32_fp64", do="mtxel", prec="fp64", n1=32, n2=32, n3=32, ecut=85.0, nv=18, nc=100, nfreq=1,
                 ng=800, ik=1, v0=0, v=18, c0=0, c=99), a=11.53, k2=1, k3=1),
        # one q-point's static self-energy of the bands around the gap
        _si(name="sigma_si24", do="sigma", prec="fp64", n1=24, n2=24, n3=24, ecut=58.0, nv=8, nc=120, ng=350, nfreq=1, ik=5, n0=4, nn=9),
        # one (k, k') block of the BSE kernel
        _si(name="bse_si24", do="bse", prec="fp64", n1=24, n2=24, n3=24, ecut=58.0, nv=8, nc=24, ng=350, nfreq=1, ik=1, jk=5, v0=1, v=7, c0=0, c=21),
        # W = eps^-1 v of every frequency of one GaSb-like q-point
        dict(_si(name="epsinv_gasb32", do="epsinv", prec="fp64", ng=800, nfreq=16, mode="W"), a=11.53),
        # all bands of one GaSb-like k-point unfolded to a symmetry-equivalent one
        dict(_si(name="unfold_gasb32", do="unfold", prec="fp64", ecut=85.0, nv=18, nb=418, fold=3), a=11.53),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["chi0", "chi0", "chi0", "mtxel", "mtxel", "bands", "noalloc", "sigma", "bse", "epsinv", "unfold"])
    c = dict(cell="fcc", a=round(rng.uniform(9.5, 12.0), 3), do=do, prec="fp64", nq=1, q1=rng.randint(0, 1), q2=0, q3=rng.randint(0, 1),
             k1=2, k2=1, k3=rng.randint(1, 3), kchunk=1, nfreq=1)
    if do == "epsinv":
        ng, nf = _log(rng, 19, 700), rng.randint(1, 16)
        return dict(c, ng=ng, nfreq=nf, mode=rng.choice(["W", "epsinv_sym", "epsinv"]))
    if do == "unfold":
        return dict(c, ecut=round(rng.uniform(12.0, 85.0), 2), nv=4, nb=_log(rng, 5, 400), fold=rng.choice([3, 4]))
    n = rng.choice(LENGTHS[:7] if do in ("sigma", "bse") else LENGTHS)
    c.update(n1=n, n2=n, n3=n)
    if do in ("mtxel", "noalloc") and rng.random() < 0.4:
        c.update(n2=rng.choice(LENGTHS), n3=rng.choice(LENGTHS))
    small = min(c["n1"], c["n2"], c["n3"])
    c["ecut"] = round(rng.uniform(0.06, 0.085) * small * small * (10.26 / c["a"]) ** 2, 3)
    share = min(1.0, (32.0 ** 3) / (c["n1"] * c["n2"] * c["n3"]))         # fewer bands on larger boxes
    c["nv"] = _log(rng, 2, 18)
    c["nc"] = max(3, int(_log(rng, 4, 260) * share))
    c["ng"] = _log(rng, 15, min(900, small ** 3 // 40))
    if do == "chi0":
        c["prec"] = rng.choice(["fp64", "mixed", "mixed", "tf32x3", "tf32"])
        c["nfreq"] = rng.randint(1, 16)
        c["nq"] = rng.choice([1, 1, 2, 3])
        c["kchunk"] = rng.randint(1, 4)
    elif do in ("mtxel", "bands"):
        c["prec"] = rng.choice(["fp64", "mixed"])
    if do in ("mtxel", "noalloc", "bse"):
        if do == "bse":
            c["nv"], c["nc"] = min(c["nv"], 10), min(c["nc"], 24)
        c.update(v0=rng.randint(0, c["nv"] - 1), c0=rng.randint(0, c["nc"] - 1))
        if do == "mtxel":          # every occupied band with a block of the empty ones, as a program short of memory walks the pairs
            c["v0"] = 0
        c.update(v=c["nv"] if do == "mtxel" else rng.randint(1, c["nv"] - c["v0"]), c=rng.randint(1, c["nc"] - c["c0"]),
                 ik=rng.randint(0, 1), jk=rng.randint(0, 1))
    if do in ("sigma", "bands"):
        nb = c["nv"] + c["nc"]
        c.update(ik=rng.randint(0, 1), n0=rng.randint(0, nb - 1))
        c["nn"] = rng.randint(1, min(12, nb - c["n0"]))
    return c


# ------------------------------------------------------------------- prepare --

def _context(case, states):
    ctx = B.bgw_create(_box(case), _kpoints(case), case["nv"], case["nc"], case["prec"])
    if case["do"] == "chi0":
        B.bgw_set_option(ctx, B.BGW_OPT_KCHUNK, case["kchunk"])
        if case["prec"] != "fp64":          # as the library's own throughput run sets them
            B.bgw_set_option(ctx, B.BGW_OPT_DEFER_K1, 1)
            B.bgw_set_option(ctx, B.BGW_OPT_OVERLAP, 1)
    else:
        for ik, (g, c, e) in enumerate(states):
            B.bgw_wfn_upload(ctx, ik, g, c, e)
    return ctx


class _State(dict):
    """A program's handles; the context is given back with the last reference."""

    def __del__(self):
        if self.get("ctx") is not None:
            B.bgw_destroy(self["ctx"])
            self["ctx"] = None


def _shift(case, ik, q):
    """k' and G0 with k_ik + q = k' + G0."""
    return _on_grid(case, _kpoints(case)[ik] + q)


def _first_q(case):
    return np.array([case["q1"] / case["k1"], case["q2"] / case["k2"], case["q3"] % case["k3"] / case["k3"]])


def _grids(case, gvec, coeff):
    """u(r) = sum_h c(h) e^{+2 pi i h.r/N} on the box, [nb][2][N1][N2][N3]."""
    n = _box(case)
    h = np.mod(gvec, np.array(n))
    idx = torch.from_numpy(((h[:, 0] * n[1] + h[:, 1]) * n[2] + h[:, 2]).astype(np.int64)).cuda()
    box = torch.zeros((*coeff.shape[:2], n[0] * n[1] * n[2]), dtype=torch.complex128, device="cuda")
    box[:, :, idx] = coeff
    return torch.fft.ifftn(box.view(*coeff.shape[:2], *n), dim=(2, 3, 4), norm="forward")


def prepare(case, seed):
    do, s = case["do"], _State(case=case)
    if do == "epsinv":
        chi, s["s"] = _polarizability(case, seed)
        s["chi"], s["out"] = chi, torch.empty_like(chi)
        s["work"] = torch.empty(B.bgw_epsinv_workspace_bytes(case["ng"], case["nfreq"]), dtype=torch.uint8, device="cuda")
        return s
    if do == "unfold":
        g, e = _sphere(case, (0.0, 0.0, 0.0), case["ecut"])
        z = _randn(_generator(seed, 0, 0), case["nb"], 2, len(g))
        z *= torch.from_numpy(1.0 / (1.0 + (3.0 * e / case["ecut"]) ** 2)).cuda()
        s["g"], s["c"], s["out"] = g, z / z.abs().square().sum((1, 2), keepdim=True).sqrt(), torch.empty_like(z)
        return s
    nb = case["nv"] + case["nc"]
    states = _states(case, seed, nb)
    cdt = torch.complex128 if case["prec"] == "fp64" else torch.complex64
    if do == "chi0":
        s["states"], s["qs"], s["freq"] = states, _qlist(case), _frequencies(case)
        s["out"] = [torch.empty((case["nfreq"], len(g), len(g)), dtype=torch.complex128, device="cuda") for _, g, _ in s["qs"]]
    elif do in ("mtxel", "bands", "noalloc"):
        s["q"] = _first_q(case)
        s["g"] = _eps_sphere(case, s["q"], case["ng"])
        rows, cols = (case["nn"], nb) if do == "bands" else (case["v"], case["c"])
        s["out"] = torch.empty((rows, cols, len(s["g"])), dtype=cdt, device="cuda")
        if do == "noalloc":
            kp, s["G0"] = _shift(case, case["ik"], s["q"])
            v, c = slice(case["v0"], case["v0"] + case["v"]), slice(case["nv"] + case["c0"], case["nv"] + case["c0"] + case["c"])
            s["Uv"] = _grids(case, states[case["ik"]][0], states[case["ik"]][1][v]).contiguous()
            s["Uc"] = _grids(case, states[kp][0], states[kp][1][c]).contiguous()
            return s
    elif do == "sigma":
        s["q"] = _first_q(case)
        s["g"] = _eps_sphere(case, s["q"], case["ng"])
        s["W"], s["v"] = _screened(case, seed, s["q"], s["g"])
    elif do == "bse":
        k = _kpoints(case)
        s["qd"], s["q0"] = k[case["jk"]] - k[case["ik"]], np.zeros(3)
        s["gd"], s["g0"] = _eps_sphere(case, s["qd"], case["ng"]), _eps_sphere(case, s["q0"], case["ng"])
        s["W"], _ = _screened(case, seed, s["qd"], s["gd"])
        s["v0"] = _coulomb(case, s["q0"], s["g0"])
        n = case["v"] * case["c"]
        s["out"] = [torch.empty((n, n), dtype=torch.complex128, device="cuda") for _ in range(2)]
    s["ctx"] = _context(case, states)
    return s


def run(s):
    case = s["case"]
    do = case["do"]
    if do == "chi0":
        B.bgw_chi0_reset(s["ctx"])
        for ik, (g, c, e) in enumerate(s["states"]):
            B.bgw_wfn_upload(s["ctx"], ik, g, c, e)
        B.bgw_chi0_accumulate(s["ctx"], s["qs"], s["freq"], 0, len(s["states"]))
        for iq, out in enumerate(s["out"]):
            B.bgw_chi0_finalize(s["ctx"], iq, out)
        return s["out"]
    if do == "mtxel":
        B.bgw_mtxel_spinor(s["ctx"], s["q"], s["g"], case["ik"], case["v0"], case["v"], case["c0"], case["c"], s["out"])
        return s["out"]
    if do == "bands":
        B.bgw_mtxel_bands(s["ctx"], s["q"], s["g"], case["ik"], case["n0"], case["nn"], 0, case["nv"] + case["nc"], s["out"])
        return s["out"]
    if do == "noalloc":
        B.bgw_mtxel_spinor_noalloc(_box(case), s["Uv"], s["Uc"], case["v"], case["c"], s["G0"], s["g"], s["out"])
        return s["out"]
    if do == "sigma":
        return B.bgw_sigma_cohsex(s["ctx"], s["q"], s["g"], case["ik"], case["n0"], case["nn"], s["W"], s["v"])
    if do == "bse":
        B.bgw_bse_kernel(s["ctx"], case["ik"], case["jk"], s["q0"], s["g0"], s["v0"], s["qd"], s["gd"], s["W"], case["v0"], case["v"],
                         case["c0"], case["c"], *s["out"])
        return s["out"]
    if do == "epsinv":
        s["out"].copy_(s["chi"])            # the call works in place
        B.bgw_epsinv(s["out"], s["s"], case["mode"], s["work"])
        return s["out"]
    _, rot, tau = _rotation(case)
    g = B.bgw_unfold_spinor(_cell(case), rot, tau, s["g"], s["c"], s["out"])
    return [s["out"], g]


# ---------------------------------------------------------------- work, exact --

def _box_flops(case):
    n = case["n1"] * case["n2"] * case["n3"]
    return n, 5.0 * n * math.log2(n)


def work(case):
    do, ng = case["do"], case.get("ng", 0)
    cb = 16 if case["prec"] == "fp64" else 8
    if do == "epsinv":
        return {"bytes": 32 * case["nfreq"] * ng * ng, "flops": 8.0 * case["nfreq"] * ng ** 3}
    if do == "unfold":
        ngw = len(_sphere(case, (0.0, 0.0, 0.0), case["ecut"])[0])
        return {"bytes": 64 * case["nb"] * ngw, "flops": 32.0 * case["nb"] * ngw}
    n, fft = _box_flops(case)
    if do == "chi0":
        nk, nb = case["k1"] * case["k2"] * case["k3"], case["nv"] + case["nc"]
        bands = sum(2 * nb * len(_sphere(case, k, case["ecut"])[0]) for k in _kpoints(case))
        out = {"bytes": 16 * bands, "flops": 2 * nk * nb * fft}
        for _, g, nc in _qlist(case):
            pairs = nk * case["nv"] * nc
            out["bytes"] += 16 * case["nfreq"] * len(g) ** 2
            out["flops"] += pairs * (16 * n + fft + 4.0 * case["nfreq"] * len(g) * (len(g) + 1))
        return out
    if do == "bse":
        v, c = case["v"], case["c"]
        pairs = 2 * v * c + v * v + c * c
        m = (v * c) ** 2
        return {"bytes": 32 * n * 2 * (v + c) + 16 * ng * ng + 32 * m,
                "flops": pairs * (16 * n + fft) + 16.0 * ng * m + 8.0 * ng * ng * v * v}
    rows, cols = {"bands": (case.get("nn"), case["nv"] + case["nc"]), "sigma": (case.get("nn"), case["nv"] + case["nc"])}.get(
        do, (case.get("v"), case.get("c")))
    out = {"bytes": 2 * cb * n * (rows + cols), "flops": rows * cols * (16 * n + fft)}
    if do == "sigma":
        out["bytes"] += 16 * ng * ng
        out["flops"] += 8.0 * rows * cols * ng * ng
    else:
        out["bytes"] += cb * rows * cols * ng
    return out


def _elements(case, uv, uc, G0, gvec):
    """M[v][c][g] by FFT of the spin-traced products, complex128."""
    n = np.array(_box(case))
    h = np.mod(gvec + np.asarray(G0)[None, :], n)
    idx = torch.from_numpy(((h[:, 0] * n[1] + h[:, 1]) * n[2] + h[:, 2]).astype(np.int64)).cuda()
    out = torch.empty((len(uv), len(uc), len(gvec)), dtype=torch.complex128, device="cuda")
    step = max(1, int(3e8 // (32 * n.prod())))
    for v in range(len(uv)):
        for c in range(0, len(uc), step):
            rho = (uv[v].conj()[None] * uc[c:c + step]).sum(1)
            out[v, c:c + step] = torch.fft.fftn(rho, dim=(1, 2, 3), norm="forward").reshape(len(rho), -1)[:, idx]
    return out


def exact(case, seed):
    do = case["do"]
    if do == "epsinv":
        chi, s = _polarizability(case, seed)
        s = torch.from_numpy(s).cuda()
        eye = torch.eye(case["ng"], dtype=torch.complex128, device="cuda")
        left, right = {"W": (s, s), "epsinv": (s, 1.0 / s), "epsinv_sym": (s / s, s / s)}[case["mode"]]
        return torch.stack([left[:, None] * torch.linalg.inv(eye - s[:, None] * c * s[None, :]) * right[None, :] for c in chi])
    if do == "unfold":
        s = prepare(case, seed)
        r, rot, tau = _rotation(case)
        theta = 2.0 * math.pi / case["fold"]
        axis = np.array([1.0, 1.0, 1.0]) / math.sqrt(3.0) if case["fold"] == 3 else np.array([0.0, 0.0, 1.0])
        x, y, z = math.sin(theta / 2) * axis
        u = torch.tensor([[math.cos(theta / 2) - 1j * z, -1j * x - y], [-1j * x + y, math.cos(theta / 2) + 1j * z]], dtype=torch.complex128, device="cuda")
        g = np.rint(s["g"] @ np.linalg.inv(rot)).astype(np.int32)
        phase = torch.from_numpy(np.exp(-2j * np.pi * (g @ tau))).cuda()
        return [torch.einsum("ab,nbg->nag", u, s["c"]) * phase, torch.from_numpy(g)]
    nb = case["nv"] + case["nc"]
    states = _states(case, seed, nb)
    nk = len(states)
    u = functools.lru_cache(maxsize=4)(lambda ik: _grids(case, states[ik][0], states[ik][1]))
    if do == "chi0":
        out = []
        for q, g, nc in _qlist(case):
            chi = torch.zeros((case["nfreq"], len(g), len(g)), dtype=torch.complex128, device="cuda")
            for ik in range(nk):
                kp, G0 = _shift(case, ik, q)
                m = _elements(case, u(ik)[:case["nv"]], u(kp)[case["nv"]:case["nv"] + nc], G0, g).reshape(-1, len(g))
                d = (states[ik][2][:case["nv"], None] - states[kp][2][None, case["nv"]:case["nv"] + nc]).reshape(-1)
                for j, w in enumerate(_frequencies(case)):
                    chi[j] += m.mH @ ((2.0 * d / (d * d + w * w))[:, None] * m)
            out.append(chi / nk)
        return out
    if do in ("mtxel", "bands", "noalloc"):
        q = _first_q(case)
        g = _eps_sphere(case, q, case["ng"])
        kp, G0 = _shift(case, case["ik"], q)
        if do == "bands":
            return _elements(case, u(case["ik"])[case["n0"]:case["n0"] + case["nn"]], u(kp), G0, g)
        v, c = slice(case["v0"], case["v0"] + case["v"]), slice(case["nv"] + case["c0"], case["nv"] + case["c0"] + case["c"])
        return _elements(case, u(case["ik"])[v], u(kp)[c], G0, g)
    if do == "sigma":
        q = _first_q(case)
        g = _eps_sphere(case, q, case["ng"])
        W, vq = _screened(case, seed, q, g)
        vq = torch.from_numpy(vq).cuda()
        kq, _ = _on_grid(case, _kpoints(case)[case["ik"]] - q)
        kp, G0 = _shift(case, kq, q)
        m = _elements(case, u(kq), u(kp)[case["n0"]:case["n0"] + case["nn"]], G0, g)
        sx = -((m[:case["nv"]].conj() @ W) * m[:case["nv"]]).sum((0, 2)).real / nk
        coh = 0.5 * (((m.conj() @ W) * m).sum((0, 2)).real - (m.abs().square() * vq).sum((0, 2))) / nk
        return sx, coh
    k = _kpoints(case)
    ik, jk, qd, q0 = case["ik"], case["jk"], k[case["jk"]] - k[case["ik"]], np.zeros(3)
    gd, g0 = _eps_sphere(case, qd, case["ng"]), _eps_sphere(case, q0, case["ng"])
    W, _ = _screened(case, seed, qd, gd)
    v0 = torch.from_numpy(_coulomb(case, q0, g0)).cuda()
    v, c = slice(case["v0"], case["v0"] + case["v"]), slice(case["nv"] + case["c0"], case["nv"] + case["c0"] + case["c"])
    n = case["v"] * case["c"]
    mi = _elements(case, u(ik)[v], u(ik)[c], (0, 0, 0), g0).reshape(n, -1)
    mj = _elements(case, u(jk)[v], u(jk)[c], (0, 0, 0), g0).reshape(n, -1)
    kp, G0 = _shift(case, ik, qd)
    cc = _elements(case, u(ik)[c], u(kp)[c], G0, gd).reshape(case["c"] ** 2, -1)
    vv = _elements(case, u(ik)[v], u(kp)[v], G0, gd).reshape(case["v"] ** 2, -1)
    kd = (cc.conj() @ W @ vv.T).reshape(case["c"], case["c"], case["v"], case["v"]).permute(2, 0, 3, 1).reshape(n, n)
    return [(mi * v0) @ mj.mH / nk, -kd / nk]
