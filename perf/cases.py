"""Performance cases of the diffuse-scattering library: what its users ask of it, by its public entry
points, from the smallest Monte-Carlo step to the largest displacive volume.

listed()        the cases by name
draw(rng)       one more case of the same ranges
prepare(c, s)   inputs of seed s on the GPU, the resident model and the output buffers
run(state)      one pass; the outputs whole
work(c)         bytes and flops of one pass that no implementation can do without
exact(c, s)     the outputs in 64 bits, from torch alone

A case is a dict of plain values.  Common keys: kind (which entry point), disorder (occ, spin,
disp), cell (a crystal of CELLS), n1 n2 n3 (supercell), nsite, nmodels, ff (form factors), mode,
precision (32, 64), hmax (|h|, |k|, |l| <= hmax on the supercell's Bragg positions), off (the grid's
start and end moved by so many Bragg positions: a grid that is not centred), seeds apart.
"""
import math

import numpy as np
import torch

import paper_1809_07088_gb300 as ds
from paper_1809_07088_gb300.autograd import diffuse_intensity

TWO_PI = 2.0 * math.pi
C_MAG = 0.07265  # barn, the constant of the magnetic intensity

FCC = [[0.0, 0.0, 0.0], [0.5, 0.5, 0.0], [0.5, 0.0, 0.5], [0.0, 0.5, 0.5]]
TET = [[0.0, 0.0, 0.0], [0.0, 0.25, 0.25], [0.25, 0.0, 0.25], [0.25, 0.25, 0.0]]
CELLS = {
    "fcc": ((4.0, 4.0, 4.0, 90.0, 90.0, 90.0), FCC),
    "pyrochlore": ((10.0, 10.0, 10.0, 90.0, 90.0, 90.0),
                   [[(a + b) % 1.0 for a, b in zip(t, v)] for t in FCC for v in TET]),
    "perovskite": ((4.0, 4.0, 4.0, 90.0, 90.0, 90.0),
                   [[0.0, 0.0, 0.0], [0.5, 0.5, 0.5], [0.5, 0.5, 0.0], [0.5, 0.0, 0.5], [0.0, 0.5, 0.5]]),
    "simple": ((4.0, 4.0, 4.0, 90.0, 90.0, 90.0), [[0.0, 0.0, 0.0]]),
    # general positions (drawn from the seed)
    "cubic": ((5.0, 5.0, 5.0, 90.0, 90.0, 90.0), None),
    "triclinic": ((4.1, 4.6, 5.2, 84.0, 97.0, 101.0), None),
}
J0 = (0.4, 15.0, 0.6, 5.0, 0.0, 1.0, 0.0, 0.0, 0.0)
FF_KIND = {"const": 0, "gauss4": 1, "j0": 2}
DIS = {"occ": ds.DS_OCC, "spin": ds.DS_SPIN, "disp": ds.DS_DISP}
MODE = {"total": ds.DS_TOTAL, "diffuse": ds.DS_DIFFUSE}
PREC = {32: ds.DS_FP32, 64: ds.DS_FP64}
EPS = 1e-8  # remainder bound of the Taylor order, unless a case says otherwise


def _case(kind, disorder, cell, n, nsite, **kw):
    c = dict(kind=kind, disorder=disorder, cell=cell, n1=n[0], n2=n[1], n3=n[2], nsite=nsite, nmodels=1,
             ff="const", mode="diffuse", precision=32, hmax=4.0, off=0)
    c.update(kw)
    return c


def listed():
    cs = [
        # a Monte-Carlo or refinement loop's smallest step: two little triclinic supercells with mixed
        # form factors, a new configuration uploaded and its volume asked for again
        ("occ_step_small", _case("volume", "occ", "triclinic", (6, 5, 4), 3, nmodels=2, ff="mixed", hmax=1.5,
                                 off=1, upload=True)),
        # the paper's ordinary supercells: nuclear diffuse and magnetic volumes of 16 pyrochlore sites
        ("occ_pyrochlore20", _case("volume", "occ", "pyrochlore", (20, 20, 20), 16, hmax=6.0)),
        ("spin_pyrochlore20", _case("volume", "spin", "pyrochlore", (20, 20, 20), 16, ff="j0", mode="total",
                                    hmax=6.0)),
        # the small displacive model in plain FP64, the path others are judged by
        ("disp_fcc8_fp64", _case("disp", "disp", "fcc", (8, 8, 8), 4, precision=64, sigma=0.1, hopen=True)),
        # an ordinary displacive volume: large |Q.u|, a high Taylor order
        ("disp_fcc32", _case("disp", "disp", "fcc", (32, 32, 32), 4, hmax=5.0, sigma=0.1)),
        # the largest model: correlated displacements, X-ray form factors, Lanczos noise reduction
        ("disp_perovskite64_lanczos", _case("disp", "disp", "perovskite", (64, 64, 64), 5, ff="gauss4", hmax=8.0,
                                            sigma=0.08, corr=3.0, eps=1e-5, lm=2, lmp=8)),
        # one step of a refinement of displacements against a target volume: forward and backward
        ("grad_fcc32", _case("grad", "disp", "fcc", (32, 32, 32), 4, mode="total", hmax=5.0, sigma=0.1)),
        # a plane off the Bragg grid, as it is plotted beside a measured (h h l) section
        ("points_hhl_plane", _case("points", "occ", "pyrochlore", (20, 20, 20), 16, hmax=5.0, np1=401, np2=401,
                                   lm=2, lmp=2)),
        # sub-box averaging of a whole volume
        ("subbox_pyrochlore20", _case("subbox", "occ", "pyrochlore", (20, 20, 20), 16, hmax=6.0, nsb=5)),
        # sub-boxes at random origins over displaced atoms on a plane
        ("subbox_points_fcc32", _case("subboxpts", "disp", "fcc", (32, 32, 32), 4, hmax=5.0, sigma=0.1, nsb=5,
                                      norigin=2516, np1=201, np2=201)),
        # moments coupled to displacements by the Debye-Waller factor
        ("spin_debye_waller", _case("volume", "spin", "pyrochlore", (20, 20, 20), 16, ff="j0", mode="total", hmax=2.0,
                                    sigma=0.05, dw=True)),
        # the serving loop: mixed requests on resident models, queued together and waited for
        ("serve_mix", _case("serve", "mix", "cubic", (0, 0, 0), 0, hmax=4.0,
                            mix="occ:16:5 spin:16:9 disp:16:3 occ:32:12 spin:32:4 disp:32:2 occ:48:7 spin:48:3")),
    ]
    return [dict(c, name=name) for name, c in cs]


SIZES = [4, 5, 6, 7, 8, 9, 10, 12, 14, 15, 16, 18, 20, 21, 24, 25, 27, 28, 30, 32, 35, 36, 40, 42, 45, 48, 49, 50, 54,
         56, 60, 63, 64]


def _size(rng, lo, hi):
    """A supercell size the library takes, spread over the logarithm of [lo, hi]."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((s for s in SIZES if lo <= s <= hi), key=lambda s: abs(math.log(s / x)))


def _cells(rng, lo, hi):
    n = _size(rng, lo, hi)
    if rng.random() < 0.5:
        return n, n, n
    return n, _size(rng, max(lo, n // 2), min(hi, 2 * n)), _size(rng, max(lo, n // 2), min(hi, 2 * n))


def _hmax(rng, n, lo, hi, most):
    """|hkl| bound in [lo, hi] whose grid has at most `most` voxels."""
    h = rng.uniform(lo, hi)
    while h > lo and np.prod([2 * round(h * x) + 1 for x in n]) > most:
        h *= 0.9
    return round(h, 2)


def draw(rng):
    kind = rng.choice(["occ", "spin", "occ", "spin", "disp", "disp", "disp64", "grad", "points", "subbox", "subboxpts",
                       "dw", "serve"])
    off = rng.choice([0, 0, 1, -3])
    if kind in ("occ", "spin"):
        n = _cells(rng, 4, 48)
        cell = rng.choice(["pyrochlore", "fcc", "perovskite", "cubic", "triclinic"])
        most = len(CELLS[cell][1]) if CELLS[cell][1] else 16
        c = _case("volume", kind, cell, n, rng.randint(1, most), hmax=_hmax(rng, n, 1.0, 6.0, 3e7), off=off,
                  ff="j0" if kind == "spin" else rng.choice(["const", "gauss4", "mixed"]),
                  mode=rng.choice(["total", "diffuse"]), precision=rng.choice([32, 32, 32, 64]),
                  nmodels=rng.choice([1, 1, 2, 3]) if n[0] <= 20 else 1)
        c["nsite"] = min(c["nsite"], 8) if c["ff"] == "gauss4" else c["nsite"]
        return dict(c, upload=rng.random() < 0.3)
    if kind == "disp":
        n = _cells(rng, 6, 40)
        cell = rng.choice(["fcc", "fcc", "perovskite", "triclinic"])
        nsite = 4 if cell == "fcc" else 5 if cell == "perovskite" else rng.randint(1, 4)
        c = _case("disp", "disp", cell, n, nsite, hmax=_hmax(rng, n, 2.0, 5.0, 3e7), off=off,
                  sigma=round(rng.uniform(0.03, 0.1), 3), mode=rng.choice(["total", "diffuse"]),
                  ff="gauss4" if cell == "perovskite" else "const", eps=rng.choice([1e-5, 1e-8]))
        if rng.random() < 0.4:
            c.update(lm=2, lmp=rng.choice([2, 4, 8]))
        return c
    if kind == "disp64":
        n = _cells(rng, 4, 10)
        return _case("disp", "disp", rng.choice(["fcc", "triclinic"]), n, rng.randint(1, 4), precision=64,
                     hmax=_hmax(rng, n, 2.0, 4.0, 4e5), sigma=round(rng.uniform(0.05, 0.1), 3), off=off)
    if kind == "grad":
        n = _cells(rng, 8, 32)
        return _case("grad", "disp", "fcc", n, 4, mode="total", hmax=_hmax(rng, n, 2.0, 5.0, 3e7), off=off,
                     sigma=round(rng.uniform(0.05, 0.1), 3))
    if kind == "points":
        n = _cells(rng, 8, 32)
        return _case("points", rng.choice(["occ", "spin"]), "pyrochlore", n, rng.randint(2, 16), ff="j0",
                     hmax=_hmax(rng, n, 2.0, 5.0, 3e7), np1=rng.randint(31, 500), np2=rng.randint(31, 500), lm=2,
                     lmp=rng.choice([2, 4]), precision=rng.choice([32, 32, 64]))
    if kind == "subbox":
        n = _cells(rng, 10, 24)
        dis = rng.choice(["occ", "occ", "spin"])
        return _case("subbox", dis, rng.choice(["pyrochlore", "triclinic"]), n,
                     rng.randint(2, 16 if dis == "occ" else 4), hmax=_hmax(rng, n, 1.0, 5.0, 1.2e7), off=off,
                     ff="j0", mode=rng.choice(["total", "diffuse"]), nsb=rng.randint(2, min(5, min(n) // 2)))
    if kind == "subboxpts":
        n = _cells(rng, 10, 32)
        dis = rng.choice(["disp", "disp", "occ", "spin"])
        return _case("subboxpts", dis, rng.choice(["fcc", "triclinic"]), n, rng.randint(1, 4), sigma=0.1, hmax=4.0,
                     nsb=rng.randint(2, 6), norigin=rng.randint(20, 2500), np1=rng.randint(20, 200),
                     np2=rng.randint(20, 200))
    if kind == "dw":
        n = _cells(rng, 8, 20)
        return _case("volume", "spin", "pyrochlore", n, rng.randint(2, 16), ff="j0", mode="total", dw=True, off=off,
                     hmax=_hmax(rng, n, 1.0, 3.0, 6e5), sigma=round(rng.uniform(0.02, 0.1), 3))
    mix = " ".join("%s:%d:%d" % (rng.choice(["occ", "spin", "disp"]), rng.choice([16, 24, 32]), rng.randint(1, 8))
                   for _ in range(rng.randint(3, 8)))
    return _case("serve", "mix", "cubic", (0, 0, 0), 0, hmax=rng.choice([2.0, 3.0, 4.0]), mix=mix)


# ---- geometry and inputs -------------------------------------------------------------------------


def _grid(c):
    """(g0, count) in supercell indices."""
    n = (c["n1"], c["n2"], c["n3"])
    g0 = tuple(-round(c["hmax"] * x) + c["off"] for x in n)
    cnt = tuple(2 * round(c["hmax"] * x) + (0 if c.get("hopen") else 1) - c["off"] % 2 for x in n)
    return g0, cnt


def _qgrid(c):
    n = (c["n1"], c["n2"], c["n3"])
    g0, cnt = _grid(c)
    return tuple(g / x for g, x in zip(g0, n)), tuple(1.0 / x for x in n), cnt


def _subcases(c):
    """The requests of a serving mix, as cases of their own."""
    out = []
    for part in c["mix"].split():
        dis, n, nsite = part.split(":")
        out.append(_case("disp" if dis == "disp" else "volume", dis, "cubic", (int(n),) * 3, int(nsite),
                         hmax=c["hmax"], mode="total" if dis == "spin" else "diffuse",
                         ff="j0" if dis == "spin" else "const", sigma=0.03))
    return out


def _crystal(c, seed):
    """(sites, b, ff kinds, ff coefficients) on the host."""
    r = np.random.RandomState(seed % (1 << 31))
    ns = c["nsite"]
    lat, sites = CELLS[c["cell"]]
    sites = r.rand(ns, 3) if sites is None else np.array(sites[:ns], dtype=np.float64)
    kind, coef = np.zeros(ns, np.int32), np.zeros((ns, 9))
    g4 = np.concatenate([r.uniform(0.5, 10.0, (ns, 4)), r.uniform(0.5, 50.0, (ns, 4)), r.uniform(0.0, 2.0, (ns, 1))], 1)
    for i in range(ns):
        k = FF_KIND[("const", "gauss4", "j0")[i % 3] if c["ff"] == "mixed" else c["ff"]]
        kind[i] = k
        coef[i] = (g4[i % 3] if c["ff"] == "mixed" else g4[i]) if k == 1 else J0 if k == 2 else 0.0
    return lat, sites, np.ones(ns), kind, coef


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _inputs(c, seed):
    """occ uint8, spins float32, disp float32 (or None) on the GPU, upload layouts."""
    g = _gen(seed * 8 + 1)
    n = (c["n1"], c["n2"], c["n3"])
    shape = (c["nmodels"], c["nsite"]) + n
    kw = dict(generator=g, device="cuda")
    occ = spins = disp = None
    if c["disorder"] == "occ":
        occ = (torch.rand(shape, **kw) < 0.3).to(torch.uint8)
    if c["disorder"] == "spin":
        # unit spins, von Mises-Fisher (kappa = 2) about one axis per site (Wood's sampler)
        axis = torch.randn((1, c["nsite"], 1, 1, 1, 3), **kw)
        axis = axis / axis.norm(dim=-1, keepdim=True)
        xi = torch.rand(shape, **kw)
        w = (1.0 + torch.log(xi + (1.0 - xi) * math.exp(-4.0)) / 2.0).clamp(-1.0, 1.0)[..., None]
        v = torch.randn(shape + (3,), **kw)
        v = v - (v * axis).sum(-1, keepdim=True) * axis
        v = v / v.norm(dim=-1, keepdim=True)
        spins = (w * axis + (1.0 - w * w).clamp_min(0.0).sqrt() * v).contiguous()
    if c["disorder"] == "disp" or c.get("dw"):
        disp = torch.randn(shape + (3,), **kw)
        if c.get("corr"):
            # white noise through a periodic Gaussian filter (in k space), rescaled to the rms
            F = torch.fft.fftn(disp, dim=(2, 3, 4))
            for a in range(3):
                k = torch.fft.fftfreq(n[a], device="cuda") * TWO_PI
                view = [1] * 6
                view[2 + a] = n[a]
                F = F * torch.exp(-0.5 * (c["corr"] * k) ** 2).view(view)
            disp = torch.fft.ifftn(F, dim=(2, 3, 4)).real
            disp = disp / disp.square().mean().sqrt()
        disp = (disp * c["sigma"]).contiguous()
    return occ, spins, disp


def _plane(c):
    """Points of an (h h l) plane, float64 [np, 3] on the GPU."""
    h = torch.linspace(-c["hmax"], c["hmax"], c["np1"], dtype=torch.float64, device="cuda")
    l = torch.linspace(-c["hmax"], c["hmax"], c["np2"], dtype=torch.float64, device="cuda")
    hh, ll = torch.meshgrid(h, l, indexing="ij")
    return torch.stack([hh, hh, ll], -1).reshape(-1, 3).contiguous()


def _origins(c, seed):
    r = np.random.RandomState((seed + 77) % (1 << 31))
    n = (c["n1"], c["n2"], c["n3"])
    o = np.zeros((c["norigin"], 4), np.int32)
    o[:, 0] = r.randint(0, c["nmodels"], c["norigin"])
    for a in range(3):
        o[:, 1 + a] = r.randint(0, n[a], c["norigin"])
    return o


def _target(c, seed):
    """A refinement's target: the closed form of independent Gaussian displacements (Laue diffuse and
    Bragg peaks), its sigma and a ripple from the seed."""
    g0, cnt = _grid(c)
    n = (c["n1"], c["n2"], c["n3"])
    lat, sites, _, _, _ = _crystal(c, seed)
    B = _recip(lat)
    sig = 0.07 * (1.0 + 0.1 * float(np.random.RandomState(seed % (1 << 31)).rand()))
    h = [torch.arange(g, g + m, device="cuda", dtype=torch.float64) / x for g, m, x in zip(g0, cnt, n)]
    q = [sum(h[a].view([-1 if i == a else 1 for i in range(3)]) * B[a, j] for a in range(3)) for j in range(3)]
    q2 = q[0] ** 2 + q[1] ** 2 + q[2] ** 2
    fall = torch.exp(-q2 * sig ** 2)
    t = 1.0 - fall
    k0 = torch.ones((1, 1, 1), dtype=torch.bool, device="cuda")
    for a in range(3):
        at = (torch.arange(g0[a], g0[a] + cnt[a], device="cuda") % n[a] == 0)
        k0 = k0 & at.view([-1 if i == a else 1 for i in range(3)])
    s = 0
    for r in sites:
        ph = 0
        for a in range(3):
            ph = ph + h[a].view([-1 if i == a else 1 for i in range(3)]) * float(r[a])
        s = s + torch.exp(2j * math.pi * ph)
    bragg = s.abs() ** 2 * fall * (n[0] * n[1] * n[2] / len(sites))
    t = torch.where(k0, t + bragg, t)
    return (t * (1.0 + 0.05 * torch.rand(t.shape, generator=_gen(seed * 8 + 3), device="cuda"))).float().contiguous()


# ---- the calls -----------------------------------------------------------------------------------

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = ds.Context(torch.cuda.current_device())
    return _ctx


class State:
    """What a user's program holds: resident models, grids, options and output buffers."""

    def __init__(self):
        self.models = []

    def __del__(self):
        for m in self.models:
            m.close()


def _model(st, c, seed, inputs):
    lat, sites, b, kind, coef = _crystal(c, seed)
    m = ds.Model(_context(), lat, sites, (c["n1"], c["n2"], c["n3"]), c["nmodels"], b, kind, coef)
    st.models.append(m)
    occ, spins, disp = inputs
    if occ is not None:
        m.upload_occupancy(occ)
    if spins is not None:
        m.upload_spins(spins)
    if disp is not None:
        m.upload_displacements(disp)
    return m


def _opts(c):
    o = dict(disorder=DIS[c["disorder"]], mode=MODE[c["mode"]], precision=PREC[c["precision"]])
    if c["disorder"] == "disp" and c["kind"] != "subboxpts":
        o.update(taylor_order=-1, taylor_eps=c.get("eps", EPS))
    if c.get("lm"):
        o.update(smoothing=ds.DS_SMOOTH_LANCZOS, lanczos_m=c["lm"], lanczos_mprime=c["lmp"])
    if c["kind"] == "subbox":
        o.update(smoothing=ds.DS_SMOOTH_SUBBOX, subbox_n=c["nsb"])
    if c["kind"] == "subboxpts":
        o.update(subbox_n=c["nsb"])
    if c.get("dw"):
        o.update(dw_coupling=1)
    return o


def prepare(case, seed):
    c = case
    st = State()
    st.kind = c["kind"]
    if c["kind"] == "serve":
        st.reqs = []
        for i, s in enumerate(_subcases(c)):
            m = _model(st, s, seed * 16 + i, _inputs(s, seed * 16 + i))
            st.reqs.append((m, _qgrid(s), torch.empty(_grid(s)[1], device="cuda"), _opts(s)))
        torch.cuda.synchronize()  # submitted work runs on the library's own streams
        return st
    dt = torch.float32 if c["precision"] == 32 else torch.float64
    inputs = _inputs(c, seed)
    st.m, st.q, st.opts = _model(st, c, seed, inputs), _qgrid(c), _opts(c)
    if c["kind"] == "grad":
        st.disp, st.target = inputs[2], _target(c, seed)
    elif c["kind"] == "points":
        st.hkl = _plane(c)
        st.out = torch.empty(st.hkl.shape[0], dtype=dt, device="cuda")
    elif c["kind"] == "subboxpts":
        st.hkl, st.origins = _plane(c), _origins(c, seed)
        st.out = torch.empty(st.hkl.shape[0], dtype=dt, device="cuda")
    else:
        st.out = torch.empty(_grid(c)[1], dtype=dt, device="cuda")
        st.up = inputs if c.get("upload") else None
    return st


def run(st):
    if st.kind == "serve":
        ctx = _context()
        tickets = [m.submit(q, out, **o) for m, q, out, o in st.reqs]
        for t in tickets:
            ctx.wait(t)
        return [r[2] for r in st.reqs]
    if st.kind == "grad":
        u = st.disp.detach().requires_grad_()
        o = st.opts
        I = diffuse_intensity(st.m, u, st.q, precision=o["precision"], taylor_eps=o["taylor_eps"])
        chi2 = (I - st.target).square().sum()
        chi2.backward()
        return {"I": I.detach(), "grad": u.grad}
    if st.kind == "points":
        return st.m.intensity_points(st.hkl, out=st.out, **st.opts)[0]
    if st.kind == "subboxpts":
        return st.m.subbox_points(st.hkl, st.origins, out=st.out, **st.opts)[0]
    if st.up is not None:
        occ, spins, _ = st.up
        if occ is not None:
            st.m.upload_occupancy(occ)
        if spins is not None:
            st.m.upload_spins(spins)
    return st.m.intensity(st.q, out=st.out, **st.opts)[0]


# ---- the work that has to be done ----------------------------------------------------------------


def _order(xmax, eps):
    """Smallest Taylor order whose remainder bound is at most eps."""
    P = 0
    while (P + 1) * math.log(max(xmax, 1e-300)) - math.lgamma(P + 2) > math.log(eps):
        P += 1
    return P


def _order_guess(c):
    """The order of Gaussian displacements of the case's sigma (the largest of so many draws)."""
    n = (c["n1"], c["n2"], c["n3"])
    q = float(np.linalg.norm(np.array([c["hmax"]] * 3) @ _recip(CELLS[c["cell"]][0])))
    big = math.sqrt(2.0 * math.log(8.0 * c["nsite"] * n[0] * n[1] * n[2]))
    return _order(q * c["sigma"] * (3.5 if c.get("corr") else big), c.get("eps", EPS))


def _work(c):
    n = (c["n1"], c["n2"], c["n3"])
    ncell, ns, nm = n[0] * n[1] * n[2], c["nsite"], c["nmodels"]
    es = 4 if c["precision"] == 32 else 8
    nvox = float(np.prod(_grid(c)[1]))
    nc = 3 if c["disorder"] == "spin" else 1
    per_atom = 1 if c["disorder"] == "occ" else 12
    data = float(nm * ns * ncell * per_atom * (2 if c.get("upload") else 1))
    fft = 2.5 * ncell * math.log2(max(2, ncell))
    zones = [min(m / x, 17.0) + 1.0 for m, x in zip(_grid(c)[1], n)]
    if c["kind"] in ("disp", "grad"):
        P = _order_guess(c)
        T = (P + 1) * (P + 2) * (P + 3) / 6
        z = [max(1.0, y - 1.0) for y in zones]
        contract = 4 * (T * z[2] + (P + 1) * (P + 2) / 2 * z[1] * z[2] + (P + 1) * z[0] * z[1] * z[2])
        flops = nm * ns * (T * (fft + 2 * ncell) + contract * ncell / 2) + 10 * nvox
        if c["kind"] == "grad":
            return dict(bytes=2 * data + 8 * nvox, flops=3 * flops)
        if c.get("lm"):
            flops += 2 * 3 * (c["lm"] * c["lmp"]) * nvox
        return dict(bytes=data + es * nvox, flops=flops)
    if c["kind"] == "subboxpts":
        # every atom's term once per point, every box summed over its cells
        npt = c["np1"] * c["np2"]
        return dict(bytes=float(data + 28 * npt), flops=float(npt) * (ns * ncell * 20 * nm + c["norigin"] * c["nsb"] ** 3 * 4 * nc))
    if c["kind"] == "subbox":
        nf = ns * nc
        return dict(bytes=data + es * nvox, flops=nf * (nf + 1) / 2 * (2 * fft + 8 * ncell) + 20 * nvox)
    if c["kind"] == "points":
        npt = c["np1"] * c["np2"]
        taps = float((2 * math.ceil(c["lm"] * c["lmp"] / 2)) ** 3)
        return dict(bytes=data + (24 + es) * npt, flops=nc * ns * fft + 2 * taps * npt + 8 * ns * nc * min(npt * taps, nvox))
    classes = 4.0 ** 3 if CELLS[c["cell"]][1] else float(np.prod(zones))
    classes = min(classes, float(np.prod(zones)))
    flops = nm * (ns * nc * fft + 4 * ns * nc * classes * ncell + 10 * nvox)
    if c.get("dw"):
        data += 12.0 * nm * ns * ncell
        flops += 2.0 * ns * nvox * 4
    return dict(bytes=data + es * nvox, flops=flops)


def work(case):
    parts = [_work(s) for s in _subcases(case)] if case["kind"] == "serve" else [_work(case)]
    return dict(bytes=float(sum(p["bytes"] for p in parts)), flops=float(sum(p["flops"] for p in parts)))


# ---- 64-bit values, from torch alone -------------------------------------------------------------


def _recip(lat):
    a, b, c = lat[:3]
    al, be, ga = (math.radians(x) for x in lat[3:])
    cx, cy = c * math.cos(be), c * (math.cos(al) - math.cos(be) * math.cos(ga)) / math.sin(ga)
    A = np.array([[a, 0, 0], [b * math.cos(ga), b * math.sin(ga), 0], [cx, cy, math.sqrt(c * c - cx * cx - cy * cy)]])
    return TWO_PI * np.linalg.inv(A).T


def _formfactor(kind, f, q2):
    s2 = q2 / (4.0 * math.pi) ** 2
    if kind == 1:
        return sum(f[i] * torch.exp(-f[4 + i] * s2) for i in range(4)) + f[8]
    if kind == 2:
        return f[0] * torch.exp(-f[1] * s2) + f[2] * torch.exp(-f[3] * s2) + f[4] * torch.exp(-f[5] * s2) + f[6]
    return torch.ones_like(s2)


def _formfactors(kind, coef, q2):
    """[nsite] list of form factors on q2, equal ones computed once."""
    seen, out = {}, []
    for k, f in zip(kind, coef):
        key = (int(k),) + (tuple(f) if k else ())
        if key not in seen:
            seen[key] = _formfactor(int(k), [float(x) for x in f], q2)
        out.append(seen[key])
    return out


def _axis(x, a, nd=3):
    v = [1] * nd
    v[a] = -1
    return x.view(v)


def _spectra(c, inputs):
    """Transforms of the request's fields, complex128 [model][site][comp][n1][n2][n3]."""
    if c["disorder"] == "occ":
        x = inputs[0].double()[:, :, None]
    else:
        x = inputs[1].double().permute(0, 1, 5, 2, 3, 4)
    if c["mode"] == "diffuse":
        x = x - x.mean(dim=(0, 3, 4, 5), keepdim=True)
    return torch.fft.ifftn(x.to(torch.complex128), dim=(3, 4, 5), norm="forward"), x


def _perp(F, Q, q2):
    """|F_perp|^2 over the leading component axis of F."""
    tot = (F.real ** 2 + F.imag ** 2).sum(0)
    par = sum(F[a] * Q[a] for a in range(3))
    safe = torch.where(q2 > 0, q2, torch.ones_like(q2))
    return torch.where(q2 > 0, tot - (par.real ** 2 + par.imag ** 2) / safe, tot * (2.0 / 3.0))


def _dw_plane(c, disp, B, h):
    """T[site][h1] -> planes [c2][c3] of the Debye-Waller factor, by products of one-axis exponentials."""
    u = disp.double()
    ut = u @ torch.tensor(B.T, device="cuda")                     # u~_a = b*_a . u
    E = []
    for s in range(c["nsite"]):
        v = ut[:, s].reshape(-1, 3)
        E.append([torch.exp(1j * v[:, a:a + 1] * h[a][None, :]) for a in range(3)])
    return lambda s, i: ((E[s][0][:, i:i + 1] * E[s][1]).T @ E[s][2]).real / E[s][0].shape[0]


def _exact_volume(c, seed, inputs, g0, cnt):
    """I(G) of occupancy or spin disorder on the grid."""
    n = (c["n1"], c["n2"], c["n3"])
    lat, sites, _, kind, coef = _crystal(c, seed)
    B = _recip(lat)
    X, _ = _spectra(c, inputs)
    ns, nc = c["nsite"], X.shape[2]
    gi = [torch.arange(g, g + m, device="cuda") for g, m in zip(g0, cnt)]
    h = [g.double() / x for g, x in zip(gi, n)]
    k = [g % x for g, x in zip(gi, n)]
    e = [torch.exp(2j * math.pi * torch.tensor(sites[:, a], device="cuda")[:, None] * h[a][None]) for a in range(3)]
    e23 = e[1][:, :, None] * e[2][:, None, :]
    dw = _dw_plane(c, inputs[2], B, h) if c.get("dw") else None
    out = torch.empty(tuple(cnt), dtype=torch.float64, device="cuda")
    N = ns * n[0] * n[1] * n[2]
    for i in range(cnt[0]):
        Q = [h[0][i] * B[0, j] + _axis(h[1], 0, 2) * B[1, j] + _axis(h[2], 1, 2) * B[2, j] for j in range(3)]
        q2 = Q[0] ** 2 + Q[1] ** 2 + Q[2] ** 2
        f = _formfactors(kind, coef, q2)
        I = 0.0
        for m in range(c["nmodels"]):
            F = torch.zeros((nc, cnt[1], cnt[2]), dtype=torch.complex128, device="cuda")
            for s in range(ns):
                amp = e23[s] * (f[s] * e[0][s, i])
                if dw:
                    amp = amp * dw(s, i)
                F += amp * X[m, s, :, k[0][i]][:, k[1]][:, :, k[2]]
            I = I + (_perp(F, Q, q2) * C_MAG if nc == 3 else F[0].real ** 2 + F[0].imag ** 2)
        out[i] = I / (c["nmodels"] * N)
    return out


class _Taylor:
    """The truncated Taylor sum over whole zones in zone order [k1][H1, H2, H3, k2, k3]."""

    def __init__(self, c, seed, disp, g0, cnt, eps):
        n = (c["n1"], c["n2"], c["n3"])
        self.c, self.n, self.g0, self.cnt = c, n, g0, cnt
        lat, self.sites, _, self.kind, self.coef = _crystal(c, seed)
        self.B = _recip(lat)
        u = disp.double()
        corners = np.array([[(g0[a] + (cnt[a] - 1) * ((b >> a) & 1)) / n[a] for a in range(3)] for b in range(8)])
        xm = float((u.reshape(-1, 3) @ torch.tensor((corners @ self.B).T, device="cuda")).abs().max())
        self.P = _order(xm, eps)
        self.H0 = [g // x for g, x in zip(g0, n)]
        self.nH = [(g + m - 1) // x - h + 1 for g, m, x, h in zip(g0, cnt, n, self.H0)]
        self.ut = u @ torch.tensor(self.B.T, device="cuda")
        H = [torch.arange(h, h + m, device="cuda").double() for h, m in zip(self.H0, self.nH)]
        k = [torch.arange(x, device="cuda").double() / x for x in n]
        g = [k[a][:, None] + H[a][None, :] for a in range(3)]                 # [k][H] r.l.u.
        self.gs = [max(abs(x) for x in (self.H0[a], self.H0[a] + self.nH[a])) for a in range(3)]
        self.g = g
        self.V = [(g[a] / self.gs[a])[..., None] ** torch.arange(self.P + 1, device="cuda") for a in range(3)]
        self.e = [[torch.exp(2j * math.pi * float(r[a]) * g[a]) for a in range(3)] for r in self.sites]

    def powers(self, m, s):
        """(gs u~)^e / e! of one site, three arrays [P + 1][n1][n2][n3]."""
        out = []
        for a in range(3):
            v, p = self.ut[m, s, ..., a] * self.gs[a], [torch.ones(self.n, dtype=torch.float64, device="cuda")]
            for e in range(1, self.P + 1):
                p.append(p[-1] * v / e)
            out.append(torch.stack(p))
        return out

    def ff(self, s, k1):
        """b f(|Q|) exp(iQ.r) of one site at [H1, H2, H3, k2, k3]."""
        g1, g2, g3 = self.g[0][k1], self.g[1], self.g[2]
        sh = [g1.view(-1, 1, 1, 1, 1), g2.T.reshape(1, -1, 1, self.n[1], 1), g3.T.reshape(1, 1, -1, 1, self.n[2])]
        e = [self.e[s][0][k1].view(-1, 1, 1, 1, 1), self.e[s][1].T.reshape(1, -1, 1, self.n[1], 1),
             self.e[s][2].T.reshape(1, 1, -1, 1, self.n[2])]
        ph = e[0] * (e[1] * e[2])
        if not self.kind[s]:
            return ph
        q2 = sum((sh[0] * self.B[0, j] + sh[1] * self.B[1, j] + sh[2] * self.B[2, j]) ** 2 for j in range(3))
        return ph * _formfactor(int(self.kind[s]), [float(x) for x in self.coef[s]], q2)

    def forward(self, m, diffuse):
        """F (minus the Bragg term: the even orders at k = 0) [k1][H1, H2, H3, k2, k3]."""
        P, n, nH, dev = self.P, self.n, self.nH, "cuda"
        V = [v.to(torch.complex128) for v in self.V]
        F = torch.zeros((n[0], nH[0], nH[1], nH[2], n[1], n[2]), dtype=torch.complex128, device=dev)
        for s in range(self.c["nsite"]):
            pw = self.powers(m, s)
            T2 = torch.empty((P + 1, nH[1], nH[2]) + tuple(n), dtype=torch.complex128, device=dev)
            even = torch.zeros((P + 1,) * 3, dtype=torch.float64, device=dev)  # k = 0 transforms, even orders
            for a in range(P + 1):
                T1 = torch.empty((P - a + 1, nH[2]) + tuple(n), dtype=torch.complex128, device=dev)
                for b in range(P - a + 1):
                    lc = P - a - b + 1
                    fld = (pw[0][a] * pw[1][b])[None] * pw[2][:lc]
                    M = torch.fft.ifftn(fld.to(torch.complex128), dim=(1, 2, 3), norm="forward")
                    if diffuse:
                        even[a, b, :lc] = M[:, 0, 0, 0].real
                    M *= _axis(torch.tensor([1j ** ((a + b + q) % 4) for q in range(lc)], device=dev), 0, 4)
                    # sum over c with x3^c, one product per k3
                    R = torch.bmm(V[2][:, :, :lc], M.permute(3, 0, 1, 2).reshape(n[2], lc, -1))
                    T1[b] = R.view(n[2], nH[2], n[0], n[1]).permute(1, 2, 3, 0)
                R = torch.bmm(V[1][:, :, :P - a + 1], T1.permute(3, 0, 1, 2, 4).reshape(n[1], P - a + 1, -1))
                T2[a] = R.view(n[1], nH[1], nH[2], n[0], n[2]).permute(1, 2, 3, 0, 4)
                del T1, R
            for k1 in range(n[0]):
                S = (V[0][k1] @ T2[:, :, :, k1].reshape(P + 1, -1)).view(nH[0], nH[1], nH[2], n[1], n[2])
                if diffuse and k1 == 0:
                    sgn = torch.tensor([(1.0, 0.0, -1.0, 0.0)[q % 4] for q in range(3 * P + 1)], dtype=torch.float64, device=dev)
                    i = torch.arange(P + 1, device=dev)
                    order = i[:, None, None] + i[None, :, None] + i[None, None, :]
                    Sb = torch.einsum("abc,xa,yb,zc->xyz", even * sgn[order], self.V[0][0], self.V[1][0], self.V[2][0])
                    S[:, :, :, 0, 0] -= Sb
                F[k1] += S * self.ff(s, k1)
            del T2
        return F

    def volume(self, F):
        """|F|^2 / N on the grid."""
        n, nH = self.n, self.nH
        I = torch.empty(F.shape, dtype=torch.float64, device="cuda")
        for k1 in range(n[0]):
            I[k1] = (F[k1].real ** 2 + F[k1].imag ** 2) / (self.c["nsite"] * n[0] * n[1] * n[2])
        I = I.permute(1, 0, 2, 4, 3, 5).reshape(nH[0] * n[0], nH[1] * n[1], nH[2] * n[2])
        o = [g - h * x for g, h, x in zip(self.g0, self.H0, n)]
        return I[o[0]:o[0] + self.cnt[0], o[1]:o[1] + self.cnt[1], o[2]:o[2] + self.cnt[2]]

    def backward(self, m, F, dLdI):
        """dL/du [site][n1][n2][n3][3] for dL/dI on the grid (one supercell, TOTAL)."""
        P, n, nH, dev = self.P, self.n, self.nH, "cuda"
        N = self.c["nsite"] * n[0] * n[1] * n[2]
        full = torch.zeros([nH[a] * n[a] for a in range(3)], dtype=torch.float64, device=dev)
        o = [g - h * x for g, h, x in zip(self.g0, self.H0, n)]
        full[o[0]:o[0] + self.cnt[0], o[1]:o[1] + self.cnt[1], o[2]:o[2] + self.cnt[2]] = dLdI
        full = full.view(nH[0], n[0], nH[1], n[1], nH[2], n[2]).permute(1, 0, 2, 4, 3, 5)
        gam = F.conj() * (full * (2.0 / N))
        V = [v.to(torch.complex128) for v in self.V]
        grad = torch.zeros((self.c["nsite"],) + tuple(n) + (3,), dtype=torch.float64, device=dev)
        for s in range(self.c["nsite"]):
            pw = self.powers(m, s)
            W = torch.empty((P + 1, nH[1], nH[2]) + tuple(n), dtype=torch.complex128, device=dev)
            for k1 in range(n[0]):
                W[:, :, :, k1] = (V[0][k1].T @ (gam[k1] * self.ff(s, k1)).reshape(nH[0], -1)).view(P + 1, nH[1], nH[2], n[1], n[2])
            gr = [0.0, 0.0, 0.0]
            for a in range(P + 1):
                nb = P - a + 1
                R = torch.bmm(V[1][:, :, :nb].transpose(1, 2), W[a].permute(3, 0, 1, 2, 4).reshape(n[1], nH[1], -1))
                T1 = R.view(n[1], nb, nH[2], n[0], n[2]).permute(1, 2, 3, 0, 4).contiguous()  # [b][H3][k1][k2][k3]
                for b in range(nb):
                    lc = P - a - b + 1
                    Z = torch.bmm(V[2][:, :, :lc].transpose(1, 2), T1[b].permute(3, 0, 1, 2).reshape(n[2], nH[2], -1))
                    Z = Z.view(n[2], lc, n[0], n[1]).permute(1, 2, 3, 0)
                    D = torch.fft.ifftn(Z, dim=(1, 2, 3), norm="forward")
                    D = (D * _axis(torch.tensor([1j ** ((a + b + q) % 4) for q in range(lc)], device=dev), 0, 4)).real
                    ab = pw[0][a] * pw[1][b]
                    dc = (D * pw[2][:lc]).sum(0)
                    if a:
                        gr[0] = gr[0] + dc * pw[0][a - 1] * pw[1][b]
                    if b:
                        gr[1] = gr[1] + dc * pw[0][a] * pw[1][b - 1]
                    if lc > 1:
                        gr[2] = gr[2] + (D[1:] * pw[2][:lc - 1]).sum(0) * ab
            for j in range(3):
                for al in range(3):
                    grad[s, ..., al] += gr[j] * (self.gs[j] * self.B[j, al])
        return grad


def _exact_disp(c, seed, inputs, g0, cnt):
    if c["nmodels"] != 1:
        return None
    t = _Taylor(c, seed, inputs[2], g0, cnt, c.get("eps", EPS))
    return t.volume(t.forward(0, c["mode"] == "diffuse"))


def _sinc(x):
    x = x * math.pi
    return torch.where(x == 0, torch.ones_like(x), torch.sin(x) / torch.where(x == 0, torch.ones_like(x), x))


def _lanczos_weight(d, lm, lmp):
    rcut, meff = (1.0 - 1.0 / lm) / lmp, 0.5 * lm * lmp
    return torch.where(d.abs() < meff, _sinc(2.0 * rcut * d) * _sinc(d / meff), torch.zeros_like(d))


def _exact_grid(c, seed, inputs, g0, cnt):
    return (_exact_disp if c["disorder"] == "disp" else _exact_volume)(c, seed, inputs, g0, cnt)


def _exact_smoothed(c, seed):
    """The requested volume, by separable passes over its halo where it is resampled."""
    inputs = _inputs(c, seed)
    g0, cnt = _grid(c)
    if not c.get("lm"):
        return _exact_grid(c, seed, inputs, g0, cnt)
    h = math.ceil(0.5 * c["lm"] * c["lmp"]) - 1
    I = _exact_grid(c, seed, inputs, tuple(g - h for g in g0), tuple(m + 2 * h for m in cnt))
    if I is None:
        return None
    w = _lanczos_weight(torch.arange(-h, h + 1, dtype=torch.float64, device="cuda"), c["lm"], c["lmp"])
    w = w / w.sum()
    for a in range(3):
        J = None
        for i in range(2 * h + 1):
            part = I.narrow(a, i, cnt[a])
            J = part * w[i] if J is None else J.add_(part, alpha=float(w[i]))
        I = J
    return I


def _exact_points(c, seed):
    inputs, hkl = _inputs(c, seed), _plane(c)
    n = (c["n1"], c["n2"], c["n3"])
    q = hkl * torch.tensor(n, dtype=torch.float64, device="cuda")
    M = math.ceil(0.5 * c["lm"] * c["lmp"])
    lo = q.floor().long()
    g0 = [int(v) - M + 1 for v in lo.min(0).values]
    cnt = [int(v) + M - g + 1 for v, g in zip(lo.max(0).values, g0)]
    I = _exact_grid(c, seed, inputs, g0, cnt)
    w, at = [], []
    for a in range(3):
        g = lo[:, a:a + 1] + torch.arange(-M + 1, M + 1, device="cuda")
        w.append(_lanczos_weight(q[:, a:a + 1] - g, c["lm"], c["lmp"]))
        at.append(g - g0[a])
    num = 0.0
    for i in range(2 * M):
        for j in range(2 * M):
            v = I[at[0][:, i:i + 1], at[1][:, j:j + 1], at[2]]
            num = num + w[0][:, i] * w[1][:, j] * (v * w[2]).sum(1)
    return num / (w[0].sum(1) * w[1].sum(1) * w[2].sum(1))


def _exact_subbox(c, seed):
    """Pair correlations windowed by the boxes' triangle, contracted voxel by voxel."""
    inputs = _inputs(c, seed)
    n = (c["n1"], c["n2"], c["n3"])
    lat, sites, _, kind, coef = _crystal(c, seed)
    B, nsb, ns = _recip(lat), c["nsb"], c["nsite"]
    X, _ = _spectra(c, inputs)
    nc = X.shape[2]
    X = X.reshape(c["nmodels"], ns * nc, *n)
    win = 1.0
    for a in range(3):
        d = torch.arange(n[a], device="cuda")
        d = torch.minimum(d, n[a] - d).double()
        win = win * _axis((nsb - d).clamp_min(0.0), a)
    S = torch.empty((ns * nc, ns * nc) + tuple(n), dtype=torch.complex128, device="cuda")
    for p in range(ns * nc):
        C = torch.fft.fftn((X[:, p:p + 1] * X.conj()).sum(0), dim=(1, 2, 3)) / (n[0] * n[1] * n[2])
        S[p] = torch.fft.ifftn(C * win, dim=(1, 2, 3), norm="forward")
    g0, cnt = _grid(c)
    gi = [torch.arange(g, g + m, device="cuda") for g, m in zip(g0, cnt)]
    h = [g.double() / x for g, x in zip(gi, n)]
    k = [g % x for g, x in zip(gi, n)]
    e = [torch.exp(2j * math.pi * torch.tensor(sites[:, a], device="cuda")[:, None] * h[a][None]) for a in range(3)]
    e23 = e[1][:, :, None] * e[2][:, None, :]
    out = torch.empty(tuple(cnt), dtype=torch.float64, device="cuda")
    for i in range(cnt[0]):
        Q = [h[0][i] * B[0, j] + _axis(h[1], 0, 2) * B[1, j] + _axis(h[2], 1, 2) * B[2, j] for j in range(3)]
        q2 = Q[0] ** 2 + Q[1] ** 2 + Q[2] ** 2
        f = torch.stack(_formfactors(kind, coef, q2))
        P = e23 * (f * e[0][:, i, None, None])                                  # [site][c2][c3]
        Sg = S[:, :, k[0][i]].index_select(2, k[1]).index_select(3, k[2])
        if nc == 1:
            out[i] = torch.einsum("pyz,qyz,pqyz->yz", P, P.conj(), Sg).real
            continue
        T = torch.einsum("pyz,qyz,paqbyz->abyz", P, P.conj(), Sg.view(ns, 3, ns, 3, *Sg.shape[2:])).real
        tr = T[0, 0] + T[1, 1] + T[2, 2]
        qq = sum(Q[a] * Q[b] * T[a, b] for a in range(3) for b in range(3))
        out[i] = C_MAG * torch.where(q2 > 0, tr - qq / torch.where(q2 > 0, q2, torch.ones_like(q2)), tr * (2.0 / 3.0))
    return out / (c["nmodels"] * n[0] * n[1] * n[2] * ns * nsb ** 3)


def _exact_subbox_points(c, seed):
    occ, spins, disp = _inputs(c, seed)
    hkl, org = _plane(c), torch.tensor(_origins(c, seed), device="cuda").long()
    n = (c["n1"], c["n2"], c["n3"])
    lat, sites, _, kind, coef = _crystal(c, seed)
    B, nsb, ns = torch.tensor(_recip(lat), device="cuda"), c["nsb"], c["nsite"]
    out = torch.empty(hkl.shape[0], dtype=torch.float64, device="cuda")
    ncell = n[0] * n[1] * n[2]
    nc = 3 if spins is not None else 1
    for s0 in range(0, hkl.shape[0], 256):
        hq = hkl[s0:s0 + 256]
        Q = hq @ B
        q2 = (Q ** 2).sum(1)
        f = _formfactors(kind, coef, q2)
        A = torch.zeros((nc, ncell * c["nmodels"], hq.shape[0]), dtype=torch.complex128, device="cuda")
        for s in range(ns):
            phi = f[s] * torch.exp(2j * math.pi * (hq @ torch.tensor(sites[s], device="cuda")))
            if disp is not None:
                x = torch.exp(1j * (disp[:, s].reshape(-1, 3).double() @ Q.T))[None]
                mean = x.real.mean(1, keepdim=True)
            else:
                x = (occ[:, s].reshape(1, -1, 1) if occ is not None else spins[:, s].reshape(-1, 3).T[:, :, None]).double()
                mean = x.mean(1, keepdim=True)
            A += phi * ((x - mean) if c["mode"] == "diffuse" else x)
        F = torch.zeros((nc, org.shape[0], hq.shape[0]), dtype=torch.complex128, device="cuda")
        for d1 in range(nsb):
            for d2 in range(nsb):
                for d3 in range(nsb):
                    cell = ((org[:, 0] * n[0] + (org[:, 1] + d1) % n[0]) * n[1] + (org[:, 2] + d2) % n[1]) * n[2] + (org[:, 3] + d3) % n[2]
                    ph = torch.exp(2j * math.pi * (hq @ torch.tensor([d1, d2, d3], dtype=torch.float64, device="cuda")))
                    F += A[:, cell] * ph
        if nc == 3:
            I = _perp(F, [Q[:, a][None] for a in range(3)], q2[None]) * C_MAG
        else:
            I = F[0].real ** 2 + F[0].imag ** 2
        out[s0:s0 + 256] = I.sum(0) / (org.shape[0] * ns * nsb ** 3)
    return out


def exact(case, seed):
    c = case
    if c["kind"] == "serve":
        return [exact(s, seed * 16 + i) for i, s in enumerate(_subcases(c))]
    if c["kind"] == "grad":
        inputs = _inputs(c, seed)
        t = _Taylor(c, seed, inputs[2], *_grid(c), c.get("eps", EPS))
        F = t.forward(0, False)
        I = t.volume(F).contiguous()
        return {"I": I, "grad": t.backward(0, F, 2.0 * (I - _target(c, seed).double()))[None]}
    if c["kind"] == "points":
        return _exact_points(c, seed)
    if c["kind"] == "subbox":
        return _exact_subbox(c, seed)
    if c["kind"] == "subboxpts":
        return _exact_subbox_points(c, seed)
    return _exact_smoothed(c, seed)
