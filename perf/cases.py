"""The work that a user of this library has it do, as cases that can be timed.

A case is a dict of plain values.  `listed` gives the standing cases, `draw`
one more of the same ranges, `prepare` what a program holds before the call
(structures on the GPU, a context), `run` one pass through the public entry
points, `work` what a pass cannot do without, and `exact` what the pass
returns, computed in 64 bits by plain torch.

Structures: rigid waters on a jittered lattice in a periodic box at the
density of the library's own box configurations, or gas-phase clusters
(O uniform in a sphere of radius 3 n^(1/3) A), random orientations, O-O at
least 2.5 A, atoms of different waters at least 1.7 A apart, multipoles drawn
per water.  Positions come in FP64, as the interface takes them.  Results of
the mixed path (FP32 pairs and grids) are handed on in single precision, as
trajectory and training files store them; those of the FP64 path in FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2201_00804_gb300 as sibfa

DEV = "cuda"
F64 = torch.float64
R_OH, HOH = 0.9572, math.radians(104.52)
CELL = 3.1035            # lattice spacing (A) of one water at 1.0 g/cm^3
TERMS = ("elec", "pen", "rep", "disp", "xdisp", "pol", "ct", "total")

# Force-field parameters (kcal/mol, A, e).
PARAMS = dict(
    ke=332.063713, debye=4.80321, d_lp=0.5, lp_half_deg=54.7356103172,
    alpha_o=1.0, alpha_h=0.5, alpha_m_damp=0.75, thole=0.28, z_o=6.0, z_h=1.0, b_o=3.0, b_h=3.4,
    cs_o=0.5, cp_o=math.sqrt(3.0) / 2.0, cs_h=1.0, cp_h=0.0, cs_lp=0.5, cp_lp=math.sqrt(3.0) / 2.0,
    g_o=1.0, g_h=0.6, nval_o=6.0, nval_h=1.0, rvdw_rep_o=1.4755, rvdw_rep_h=1.10, rvdw_rep_lp=1.30,
    rep_alpha=14.0, rep_alpha2=16.3333, rep_c1=93884.0, rep_c2=46942.0, rep_f=0.8, occ_bond=2.0, n_lp=2.0,
    rvdw_disp_o=1.2594, rvdw_disp_h=0.95, rvdw_disp_lp=0.9042, disp_alpha=1.2, beta_o=1.0, beta_h=0.45,
    c6=0.5459, c8=0.4453, c10=0.3591, gamma6=2.0, gamma8=2.3, gamma10=2.6, disp_delta=0.30,
    xd_c1=20.0, xd_a1=4.5, xd_c2=8.0, xd_a2=4.5, xd_c3=10.0, xd_a3=4.5,
    ct_eta=2.2, ct_t=0.3944, ct_m=0.3133, ct_ae=2000.0, ct_ah=60.0, rvdw_ct_o=1.50, rvdw_ct_h=1.10)


def _box(name, do, sides, *, n_mol=0, edge=CELL, rc=9.0, grid=(0, 0, 0), tol=1e-6, precision="mixed", **more):
    """A periodic box of sides[0] x sides[1] x sides[2] lattice cells, n_mol of them filled (0: all)."""
    c = dict(name=name, do=do, nx=sides[0], ny=sides[1], nz=sides[2], n_mol=n_mol or sides[0] * sides[1] * sides[2],
             lx=sides[0] * edge, ly=sides[1] * edge, lz=sides[2] * edge, rc=rc, tol=tol, precision=precision, **more)
    for k, g, l in zip("xyz", grid, (c["lx"], c["ly"], c["lz"])):
        c["k" + k] = g or _smooth(1.3 * l)
    return c


def _smooth(x):
    """Smallest grid size >= x with no prime factor above 5."""
    n = max(8, math.ceil(x))
    while True:
        m = n
        for f in (2, 3, 5):
            while m % f == 0:
                m //= f
        if m == 1:
            return n
        n += 1


def listed():
    return [
        # one small gas-phase cluster: a single-point energy and force call where launches and latency count
        dict(name="cluster8", do="evaluate", clusters=1, n_min=8, n_max=8, tol=1e-6, precision="mixed"),
        # a short list of clusters in FP64, with the terms of each: reference data for a fit
        dict(name="clusters48_fp64", do="clusters", clusters=48, n_min=2, n_max=32, tol=1e-8, precision="fp64"),
        # the cluster workload: thousands of clusters of 2-32 waters in one context
        dict(name="clusters4096", do="evaluate", clusters=4096, n_min=2, n_max=32, tol=1e-6, precision="mixed"),
        # the smallest periodic box, mixed precision and tight dipoles
        _box("water216", "evaluate", (6, 6, 6), edge=18.62 / 6, rc=7.0, grid=(24, 24, 24), tol=1e-8),
        # the same in FP64: the accuracy reference
        _box("water216_fp64", "evaluate", (6, 6, 6), edge=18.62 / 6, rc=7.0, grid=(24, 24, 24), tol=1e-8,
             precision="fp64"),
        # induced dipoles alone (a property run) in an orthorhombic, not quite full box
        _box("dipoles971", "dipoles", (9, 10, 11), n_mol=971),
        # one structure of the 4096-water box: energy and forces
        _box("water4096", "evaluate", (16, 16, 16), edge=49.66 / 16, grid=(64, 64, 64)),
        # a constant-pressure step on an uneven box: energy, forces and virial
        _box("virial2028", "virial", (12, 13, 13)),
        # a served MD job on the 4096-water box: two relaxation steps, then ten steps of dynamics
        _box("md4096", "md", (16, 16, 16), edge=49.66 / 16, grid=(64, 64, 64), steps=10),
        # one structure of the 32,000-water box: the largest single call
        _box("water32000", "evaluate", (32, 32, 32), n_mol=32000, edge=98.6 / 32, grid=(108, 108, 108)),
        # dynamics of the 32,000-water box, the headline workload
        _box("md32000", "md", (32, 32, 32), n_mol=32000, edge=98.6 / 32, grid=(108, 108, 108), steps=10),
    ]


def draw(rng):
    """One more case of these ranges: clusters (1 to 4096 of 2 to 32 waters, or one of up to 256) and boxes of
    216 to 32,000 waters of any shape, calls and precisions as listed (FP64 up to about 1000 waters)."""
    log = lambda a, b: math.exp(rng.uniform(math.log(a), math.log(b)))  # noqa: E731
    fp64 = rng.random() < 0.2
    if rng.random() < 0.35:
        if rng.random() < 0.3:
            n = round(log(2, 256))
            return dict(do="evaluate", clusters=1, n_min=n, n_max=n, tol=1e-6, precision="fp64" if fp64 else "mixed")
        lo = rng.randint(2, 16)
        return dict(do="clusters" if rng.random() < 0.3 else "evaluate", clusters=round(log(8, 64 if fp64 else 4096)),
                    n_min=lo, n_max=rng.randint(lo, 32), tol=1e-6, precision="fp64" if fp64 else "mixed")
    do = "evaluate" if fp64 else rng.choice(["evaluate", "evaluate", "dipoles", "virial", "md"])
    side = log(6, 10 if fp64 else 30)
    sides = tuple(max(6, round(side + rng.uniform(-1, 1))) for _ in range(3))
    full = sides[0] * sides[1] * sides[2]
    c = _box("", do, sides, n_mol=full - rng.randint(0, full // 50), rc=9.0 if min(sides) > 6 else 7.0,
             tol=1e-8 if fp64 else 1e-6, precision="fp64" if fp64 else "mixed")
    del c["name"]
    if do == "md":
        c["steps"] = rng.randint(2, 10)
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _sizes(case):
    """Sizes of a case's clusters: the case's own, whatever the seed."""
    return np.random.default_rng(case["clusters"]).integers(case["n_min"], case["n_max"] + 1, size=case["clusters"])


def _n_mol(case):
    return int(_sizes(case).sum()) if "clusters" in case else case["n_mol"]


def _orient(shape, gen):
    """Waters (O at the origin) in uniform random orientations: (*shape, 3, 3)."""
    u = torch.rand((*shape, 3), generator=gen, device=DEV, dtype=F64)
    a, b = torch.sqrt(1 - u[..., 0]), torch.sqrt(u[..., 0])
    p, s = 2 * math.pi * u[..., 1], 2 * math.pi * u[..., 2]
    w, x, y, z = a * torch.sin(p), a * torch.cos(p), b * torch.sin(s), b * torch.cos(s)
    # images of the body's x and z axes
    ex = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + z * w), 2 * (x * z - y * w)], -1)
    ez = torch.stack([2 * (x * z + y * w), 2 * (y * z - x * w), 1 - 2 * (x * x + y * y)], -1)
    sx, cz = R_OH * math.sin(HOH / 2), R_OH * math.cos(HOH / 2)
    return torch.stack([torch.zeros_like(ex), sx * ex + cz * ez, cz * ez - sx * ex], -2)


def _clash(d):
    """Whether waters with atom-atom displacements d (..., 3, 3, 3) are too close."""
    r2 = d.square().sum(-1)
    return (r2[..., 0, 0] < 2.5 ** 2) | (r2.flatten(-2).amin(-1) < 1.7 ** 2)


def _box_positions(case, gen):
    n = (case["nx"], case["ny"], case["nz"])
    box = torch.tensor([case["lx"], case["ly"], case["lz"]], device=DEV, dtype=F64)
    ax = [torch.arange(k, device=DEV, dtype=F64) for k in n]
    centre = (torch.stack(torch.meshgrid(*ax, indexing="ij"), -1) + 0.5) * (box / torch.tensor(n, device=DEV))
    there = torch.ones(n[0] * n[1] * n[2], device=DEV, dtype=torch.bool)
    there[torch.randperm(there.numel(), generator=gen, device=DEV)[case["n_mol"]:]] = False
    there = there.view(n)
    half = [(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1) if (i, j, k) > (0, 0, 0)]
    x, redo = None, there
    for _ in range(200):
        o = centre + 0.8 * (torch.rand((*n, 3), generator=gen, device=DEV, dtype=F64) - 0.5)
        new = o[..., None, :] + _orient(n, gen)
        x = new if x is None else torch.where(redo[..., None, None], new, x)
        redo = torch.zeros_like(there)
        for s in half:
            d = torch.roll(x, s, (0, 1, 2))[..., None, :, :] - x[..., :, None, :]
            d = d - box * torch.round(d / box)
            redo |= _clash(d) & there & torch.roll(there, s, (0, 1, 2))
        if not bool(redo.any()):
            break
    return x[there]


def _cluster_positions(case, gen):
    size = torch.tensor(_sizes(case), device=DEV)
    n = int(size.max())
    real = torch.arange(n, device=DEV)[None] < size[:, None]
    lower = torch.ones((n, n), device=DEV, dtype=torch.bool).tril(-1)
    x, redo = None, real
    for _ in range(200):
        u = torch.randn((*real.shape, 3), generator=gen, device=DEV, dtype=F64)
        r = 3.0 * (size[:, None] * torch.rand(real.shape, generator=gen, device=DEV, dtype=F64)) ** (1 / 3)
        new = (u * (r / u.norm(dim=-1))[..., None])[..., None, :] + _orient(real.shape, gen)
        x = new if x is None else torch.where(redo[..., None, None], new, x)
        redo = torch.zeros_like(real)
        for part in torch.split(torch.arange(real.shape[0], device=DEV), 512):
            y, ok = x[part], real[part]
            d = y[:, :, None, :, None, :] - y[:, None, :, None, :, :]
            redo[part] = (_clash(d) & lower & ok[:, :, None] & ok[:, None, :]).any(-1)
        if not bool(redo.any()):
            break
    return x[real]


def _multipoles(m, rng):
    """Local-frame multipoles (q, mu, Theta) of m waters on O, H1, H2 and the two bond midpoints."""
    mp = np.zeros((m, 5, 10))
    mp[:, 0, 0] = rng.uniform(-0.85, -0.75, m)
    mp[:, 1:, 0] = -mp[:, :1, 0] / 4
    lo, hi = np.array([0.0, 0.0, 0.0, -0.1, -0.1]), np.array([0.3, 0.1, 0.1, 0.1, 0.1])
    mp[:, :, 3] = rng.uniform(lo, hi, (m, 5))
    th = rng.uniform(-1, 1, (m, 5, 3)) * np.array([0.5, 0.1, 0.1, 0.2, 0.2])[:, None]
    mp[:, :, 4:7] = th - th.mean(-1, keepdims=True)
    return mp


def _inputs(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    x = (_cluster_positions if "clusters" in case else _box_positions)(case, gen)
    return x, _multipoles(x.shape[0], np.random.default_rng(seed))


class _Context:
    """A library context that is given back when the program drops it."""

    def __init__(self, case, mp):
        kw = dict(precision=sibfa.PREC_FP64 if case["precision"] == "fp64" else sibfa.PREC_MIXED,
                  pcg_tol_D=case["tol"], periodic="clusters" not in case,
                  # separate structures start from the direct field; a trajectory extrapolates its own dipoles
                  warm_start=5 if case["do"] == "md" else 0)
        if kw["periodic"]:
            kw.update(box=(case["lx"], case["ly"], case["lz"]), rc=case["rc"],
                      grid=(case["kx"], case["ky"], case["kz"]), ewald_alpha=0.4)
        elif case["clusters"] > 1:
            kw["cluster_start"] = np.concatenate([[0], np.cumsum(_sizes(case))])
        self.handle = sibfa.sibfa_create(PARAMS, mp, **kw)

    def __del__(self):
        if getattr(self, "handle", None):
            sibfa.sibfa_destroy(self.handle)


def prepare(case, seed):
    x, mp = _inputs(case, seed)
    s = dict(case=case, ctx=_Context(case, mp), pos=x.reshape(-1).contiguous())
    if case["do"] == "dipoles":
        s["mu"] = torch.zeros_like(s["pos"])
    elif case["do"] == "md":
        m = torch.tensor([15.999, 1.008, 1.008], device=DEV, dtype=F64).repeat(x.shape[0])
        gen = torch.Generator(device=DEV).manual_seed(seed + 1)
        v = torch.randn((m.numel(), 3), generator=gen, device=DEV, dtype=F64)
        s["masses"] = m
        s["vel"] = (v * torch.sqrt(0.0019872041 * 300.0 * 4.184e-4 / m)[:, None]).reshape(-1)
    else:
        s["forces"] = torch.zeros_like(s["pos"])
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _hand_on(t, case):
    return t if case["precision"] == "fp64" else t.float() if torch.is_tensor(t) else t.astype(np.float32)


def run(s):
    case, ctx = s["case"], s["ctx"].handle
    if case["do"] == "dipoles":
        sibfa.sibfa_solve_dipoles(ctx, s["pos"], s["mu"])
        return {"mu": _hand_on(s["mu"], case)}
    if case["do"] == "md":
        # a job: the arrived structure relaxed, then run
        pos, vel = s["pos"].clone(), s["vel"].clone()
        sibfa.sibfa_minimize(ctx, pos, 2)
        e = sibfa.sibfa_md_steps(ctx, pos, vel, s["masses"], 0.5, case["steps"])
        return {"terms": e, "pos": _hand_on(pos, case), "vel": _hand_on(vel, case)}
    if case["do"] == "virial":
        w = np.zeros((3, 3))
        e = sibfa.sibfa_energy_forces(ctx, s["pos"], s["forces"], virial=w)
        return {"terms": e, "forces": _hand_on(s["forces"], case), "virial": _hand_on(w, case)}
    e = sibfa.sibfa_energy_forces(ctx, s["pos"], s["forces"])
    out = {"terms": e, "forces": _hand_on(s["forces"], case)}
    if case["do"] == "clusters":
        t = sibfa.sibfa_cluster_terms(ctx, case["clusters"])
        out["clusters"] = _hand_on(np.array([[d[k] for k in TERMS] for d in t]), case)
    return out


def work(case):
    """Bytes: positions, multipoles and the results once.  Operations: those of the formulas per molecule pair
    inside the cutoff, each pair once, and per grid pass and iteration of the dipole solve."""
    m = _n_mol(case)
    if "clusters" in case:
        n = _sizes(case).astype(np.float64)
        pairs, grid = float((n * (n - 1) / 2).sum()), 0.0
    else:
        volume = case["lx"] * case["ly"] * case["lz"]
        pairs = m * (m / volume) * (4.0 / 3.0) * math.pi * case["rc"] ** 3 / 2
        grid = float(case["kx"] * case["ky"] * case["kz"])
    fft = 5.0 * grid * math.log2(grid) if grid else 0.0
    iters = 12 if case["tol"] <= 1e-8 else 8
    spme = lambda sites: (2 * 125 * 20 * sites * m + 2 * fft + 2 * grid if grid else 0.0)  # noqa: E731
    # 25 multipole site pairs of 300; 4 bond-bond, 8 bond-lone pair and 4 lone pair items of 850, 455 and 220;
    # 25 dispersion point pairs of 70; 8 charge-transfer pairs of 100; 9 induced pairs of 30 per product
    solve = iters * (pairs * 9 * 30 + spme(3))
    field = pairs * 25 * 150 + spme(5)
    full = pairs * (25 * 300 + 4 * 850 + 8 * 455 + 4 * 220 + 25 * 70 + 8 * 100 + 34 * 150) + 3 * spme(5) + solve
    times = case["steps"] + 3 if case["do"] == "md" else 1
    moved = {"md": 4, "dipoles": 2}.get(case["do"], 2)
    return {"bytes": m * (400.0 + 72.0 * moved), "flops": times * (field + solve if case["do"] == "dipoles" else full)}


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch.  Sites of a water: O, H1, H2, the two
# bond midpoints, then the two lone pairs.  Gradients by reverse mode with
# respect to the sites, dipoles and quadrupoles, then through their geometry.
# ---------------------------------------------------------------------------
P = PARAMS
ZN = (P["z_o"], P["z_h"], P["z_h"], 0.0, 0.0)
BN = (P["b_o"], P["b_h"], P["b_h"], 0.0, 0.0)
ALPHA = (P["alpha_o"], P["alpha_h"], P["alpha_h"], P["alpha_m_damp"], P["alpha_m_damp"])
EW = 0.4


def _vec(*v):
    return torch.tensor(v, device=DEV, dtype=F64)


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _axes(z, x):
    z = _unit(z)
    x = _unit(x - (x * z).sum(-1, keepdim=True) * z)
    return torch.stack([x, torch.linalg.cross(z, x, dim=-1), z], -1)


def _geometry(x, mp):
    """Points (M, 7, 3), dipoles (M, 5, 3) and quadrupoles (M, 5, 3, 3) of the waters at x (M, 3, 3)."""
    o, h1, h2 = x.unbind(1)
    f0 = _axes(_unit(h1 - o) + _unit(h2 - o), h1 - o)
    f1, f2 = _axes(o - h1, h2 - h1), _axes(o - h2, h1 - h2)
    f = torch.stack([f0, f1, f2, f1, f2], 1)
    t = math.radians(P["lp_half_deg"])
    back, side = -math.cos(t) * P["d_lp"] * f0[..., 2], math.sin(t) * P["d_lp"] * f0[..., 1]
    pts = torch.stack([o, h1, h2, 0.5 * (o + h1), 0.5 * (o + h2), o + back + side, o + back - side], 1)
    th = mp[..., [4, 7, 8, 7, 5, 9, 8, 9, 6]].view(*mp.shape[:2], 3, 3)
    return pts, (f @ mp[..., 1:4, None])[..., 0], f @ th @ f.mT


def _erfc_kernel(r, n):
    """g_0..g_n of erfc(a r)/r, g_{k+1} = g_k' / r."""
    g, e = [torch.erfc(EW * r) / r], torch.exp(-(EW * r) ** 2) * 2 * EW / math.sqrt(math.pi)
    for k in range(n):
        g.append(-((2 * k + 1) * g[-1] + (-2 * EW * EW) ** k * e) / r ** 2)
    return g


def _bare_kernel(r, n):
    g = [1 / r]
    for k in range(n):
        g.append(-(2 * k + 1) * g[-1] / r ** 2)
    return g


def _exp_kernel(r, b, n):
    """g_0..g_2 of exp(-b r)/r."""
    e = torch.exp(-b * r) / r
    return [e, -e * (1 + b * r) / r ** 2, e * (3 + 3 * b * r + (b * r) ** 2) / r ** 4][: n + 1]


def _thole_kernel(r, au, periodic, n):
    """g_1..g_n damped by Thole's exponential for polarizability products au = alpha alpha' (g_0 is not used)."""
    t = P["thole"] * r ** 3 / torch.sqrt(au)
    e = torch.exp(-t)
    cut = [e, (1 + t) * e, (1 + t + 0.6 * t * t) * e]
    bare = _bare_kernel(r, n)
    base = _erfc_kernel(r, n) if periodic else bare
    return [None] + [base[k] - cut[k - 1] * bare[k] for k in range(1, n + 1)]


def _dot(a, b):
    return (a * b).sum(-1)


def _field(x, g, mu, th, q=None, second=False):
    """Potential (None where g_0 is not given), its gradient and, on request, a function for the contraction of
    its second derivatives, of a multipole at displacement x (to the target) through the kernels g."""
    tx = (th @ x[..., None])[..., 0] if th is not None else 0 * x
    s, w = _dot(mu, x), _dot(x, tx)
    phi = None
    if g[0] is not None:
        phi = w * g[2] / 3 - s * g[1] + (0 if q is None else q * g[0])
    if len(g) < 4:
        return phi, None, None
    a = w * g[3] / 3 - s * g[2] + (0 if q is None else q * g[1])
    grad = a[..., None] * x - g[1][..., None] * mu + (2 / 3) * g[2][..., None] * tx
    if not second:
        return phi, grad, None
    b = w * g[4] / 3 - s * g[3] + (0 if q is None else q * g[2])
    u = -g[2][..., None] * mu + (2 / 3) * g[3][..., None] * tx

    def contract(t):   # traceless t : second derivatives
        tx2 = (t @ x[..., None])[..., 0]
        both = (t * th).sum((-1, -2))
        return b * _dot(x, tx2) + 2 * _dot(u, tx2) + (2 / 3) * g[2] * both

    return phi, grad, contract


class _Pairs:
    """The molecule pairs i < j of a case and the shift of j's image, in pieces."""

    def __init__(self, x, case):
        o = x[:, 0]
        self.periodic = "clusters" not in case
        idx = torch.arange(o.shape[0], device=DEV)
        found, shift = [], []
        if self.periodic:
            box = _vec(case["lx"], case["ly"], case["lz"])
            for part in torch.split(idx, max(1, 20_000_000 // o.shape[0])):
                d = o[None] - o[part, None]
                sh = -box * torch.round(d / box)
                k = (((d + sh).square().sum(-1) < (case["rc"] + 2.6) ** 2) & (idx[None] > part[:, None])).nonzero()
                found.append(torch.stack([part[k[:, 0]], k[:, 1]], -1))
                shift.append(sh[k[:, 0], k[:, 1]])
            self.rc = case["rc"]
        else:
            size = torch.tensor(_sizes(case), device=DEV)
            of = torch.repeat_interleave(torch.arange(size.numel(), device=DEV), size)
            last = torch.cumsum(size, 0)[of]
            span = torch.arange(1, int(size.max()) + 1, device=DEV)
            k = (idx[:, None] + span < last[:, None]).nonzero()
            found.append(torch.stack([k[:, 0], k[:, 0] + 1 + k[:, 1]], -1))
            shift.append(torch.zeros((k.shape[0], 3), device=DEV, dtype=F64))
            self.rc = math.inf
        self.ij, self.shift = torch.cat(found), torch.cat(shift)

    def __iter__(self):
        for part in torch.split(torch.arange(self.ij.shape[0], device=DEV), 40_000):
            i, j = self.ij[part].unbind(-1)
            yield i, j, self.shift[part][:, None]


def _charges_pair(pair, per, a, b):
    """Multipole and penetration energy of each molecule pair; a, b: (points, q, mu, th)."""
    xa, qa, ma, ta = a[0][:, :5, None], a[1][:, :, None], a[2][:, :, None], a[3][:, :, None]
    xb, qb, mb, tb = b[0][:, None, :5], b[1][:, None], b[2][:, None], b[3][:, None]
    x = xa - xb
    r = x.norm(dim=-1)
    inside = (r < pair.rc).to(F64)
    ma, ta, mb, tb = (t.expand(*x.shape[:3], *t.shape[3:]) for t in (ma, ta, mb, tb))
    phi, grad, second = _field(x, _erfc_kernel(r, 4) if per else _bare_kernel(r, 4), mb, tb, qb, True)
    elec = qa * phi + _dot(ma, grad) + second(ta) / 3
    z, bn = _vec(*ZN), _vec(*BN)
    atom = (z > 0).to(F64)
    na, nb = ((z - a[1]) * atom)[:, :, None], ((z - b[1]) * atom)[:, None]
    ea, eb = torch.exp(-bn[:, None] * r), torch.exp(-bn[None] * r)
    pen = (qa * nb * eb + qb * na * ea + na * nb * ea * eb) / r
    pen = pen + na * _field(x, _exp_kernel(r, bn[:, None], 2), mb, tb)[0]
    pen = pen + nb * _field(-x, _exp_kernel(r, bn[None], 2), ma, ta)[0]
    return P["ke"] * (elec * inside).sum((1, 2)), P["ke"] * (pen * inside).sum((1, 2))


def _cos(u, v):
    return _dot(u, v) / (u.norm(dim=-1) * v.norm(dim=-1))


def _repulsion_pair(pair, a, b):
    """Exchange-repulsion of each molecule pair: overlaps of bonds and lone pairs."""
    f = P["rep_f"]
    cs, cp = (P["cs_o"], P["cs_h"], P["cs_lp"]), (P["cp_o"], P["cp_h"], P["cp_lp"])
    rv, g = (P["rvdw_rep_o"], P["rvdw_rep_h"], P["rvdw_rep_lp"]), (P["g_o"], P["g_h"], P["g_o"])
    cl = 1 - P["n_lp"] / P["nval_o"]

    def orbitals(w):
        """Four orbitals (two bonds, two lone pairs): centre, occupation and its atoms (kind, place, p axis, factor)."""
        x, q = w[0], w[1]
        co = 1 - q[:, 0] / P["nval_o"]
        out = []
        for k in (1, 2):
            ax = x[:, k] - x[:, 0]
            out.append((0.5 * (x[:, 0] + x[:, k]), P["occ_bond"],
                        [(0, x[:, 0], ax, co), (1, x[:, k], -ax, 1 - q[:, k] / P["nval_h"])]))
        for k in (5, 6):
            out.append((x[:, k], P["n_lp"], [(2, x[:, 0], x[:, k] - x[:, 0], torch.full_like(co, cl))]))
        return out

    total = 0
    for c1, n1, at1 in orbitals(a):
        for c2, n2, at2 in orbitals(b):
            lp1, lp2 = len(at1) == 1, len(at2) == 1
            pp = f if lp1 != lp2 else 2.0
            o1 = o2 = 0
            for k1, x1, p1, f1 in at1:
                for k2, x2, p2, f2 in at2:
                    v = x2 - x1
                    # two lone pairs: the angles look at the other lone pair
                    u1 = _cos(p1, c2 - x1 if lp1 and lp2 else v)
                    u2 = _cos(p2, c1 - x2 if lp1 and lp2 else -v)
                    s = cs[k1] * cs[k2] + f * (cs[k2] * cp[k1] * u1 + cs[k1] * cp[k2] * u2) + pp * cp[k1] * cp[k2] * u1 * u2
                    s = s * torch.sqrt(g[k1] * g[k2] * f1 * f2)
                    rho = v.norm(dim=-1) / (4 * math.sqrt(rv[k1] * rv[k2]))
                    o1 = o1 + s * torch.exp(-P["rep_alpha"] * rho)
                    o2 = o2 + s * torch.exp(-P["rep_alpha2"] * rho)
            r = (c1 - c2).norm(dim=-1)
            total = total + n1 * n2 * (P["rep_c1"] * o1 ** 2 / r + P["rep_c2"] * o2 ** 2 / r ** 2) * (r < pair.rc)
    return total


def _dispersion_pair(pair, a, b):
    """Dispersion and exchange-dispersion of each molecule pair over O, H1, H2 and the lone pairs."""
    at = [0, 1, 2, 5, 6]
    rv = _vec(P["rvdw_disp_o"], P["rvdw_disp_h"], P["rvdw_disp_h"], P["rvdw_disp_lp"], P["rvdw_disp_lp"])
    beta = _vec(P["beta_o"], P["beta_h"], P["beta_h"], P["beta_o"], P["beta_o"])
    nval = _vec(P["nval_o"], P["nval_h"], P["nval_h"], P["nval_o"], P["nval_o"])
    n = P["n_lp"]
    r = (a[0][:, at, None] - b[0][:, None, at]).norm(dim=-1)
    m = r / (2 * torch.sqrt(rv[:, None] * rv))
    d = (rv[:, None] + rv) * P["disp_alpha"] / r - 1
    e = sum(P["c%d" % k] * torch.exp(-P["gamma%d" % k] * d) / m ** k for k in (6, 8, 10))
    lone = torch.tensor([0, 0, 0, 1, 1], device=DEV)
    kind = lone[:, None] + lone
    weight = torch.where(kind == 0, -beta[:, None] * beta, _vec(0.0, -P["disp_delta"] / 2, -n * n / 4)[kind])
    xd = _vec(P["xd_c1"], n / 2 * P["xd_c3"], n * n / 4 * P["xd_c2"])[kind] * torch.exp(
        -_vec(P["xd_a1"], P["xd_a3"], P["xd_a2"])[kind] * m)
    ca, cb = (beta * (1 - w[1][:, [0, 1, 2, 0, 0]] / nval) for w in (a, b))
    inside = (r < pair.rc).to(F64)
    return (weight * e * inside).sum((1, 2)), (ca[:, :, None] * cb[:, None] * xd * inside).sum((1, 2))


def _transfer_pair(pair, d, a, v, vint):
    """Charge transfer from the lone pairs of d (potentials v) to the bonds of a (own potentials vint)."""
    c, lone = d[0][:, None, None, 0], d[0][:, 5:, None]
    o, h = a[0][:, None, None, 0], a[0][:, None, 1:3]
    v = v[:, :, None]

    def part(x, vi, rv):
        w = torch.exp(-P["ct_eta"] * (x - c).norm(dim=-1) / (2 * math.sqrt(P["rvdw_ct_o"] * rv)))
        return w * (vi - v) * (P["cs_lp"] * P["ct_t"] + P["cp_lp"] * P["ct_m"] * _cos(lone - c, x - c))

    e = part(o, vint[:, None, :1], P["rvdw_ct_o"]) - part(h, vint[:, None, 1:], P["rvdw_ct_h"])
    e = -P["n_lp"] * e ** 2 / (P["ct_ae"] + v - P["ct_ah"])
    return e.sum((1, 2)) * ((o - c)[:, 0, 0].norm(dim=-1) < pair.rc)


class _Grid:
    """Smooth particle mesh Ewald of order 5: charge grids of point multipoles and their convolution."""

    def __init__(self, case):
        self.k = (case["kx"], case["ky"], case["kz"])
        self.box = _vec(case["lx"], case["ly"], case["lz"])
        self.per = _vec(*self.k) / self.box
        m4 = _vec(1, 11, 11, 1) / 24
        mod, freq = [], []
        for n, l in zip(self.k, self.box):
            ph = 2 * math.pi * torch.arange(n, device=DEV, dtype=F64)[:, None] * _vec(0, 1, 2, 3) / n
            den = (m4 * torch.cos(ph)).sum(-1) ** 2 + (m4 * torch.sin(ph)).sum(-1) ** 2
            near = 0.5 * (torch.roll(den, 1) + torch.roll(den, -1))
            mod.append(1 / torch.where(den < 1e-7, near, den))
            i = torch.arange(n, device=DEV)
            freq.append(torch.where(i > n // 2, i - n, i) / l)
        m2 = freq[0][:, None, None] ** 2 + freq[1][:, None] ** 2 + freq[2] ** 2
        g = P["ke"] * torch.exp(-math.pi ** 2 * m2 / EW ** 2) / (math.pi * self.box.prod() * m2)
        g = g * mod[0][:, None, None] * mod[1][:, None] * mod[2] * math.prod(self.k)
        g[0, 0, 0] = 0
        self.g = g

    def spread(self, x, q, mu, th):
        """Grid of the multipoles at x (N, 3); q, mu, th may be None."""
        u = x * self.per
        base = torch.floor(u.detach())
        w = u - base

        def spline(n):   # M_n at w + j, j = 0..n-1
            b = [w, 1 - w]
            for o in range(3, n + 1):
                b = [((w + j) * (b[j] if j < o - 1 else 0) + (o - w - j) * (b[j - 1] if j else 0)) / (o - 1)
                     for j in range(o)]
            return b

        zero = torch.zeros_like(w)
        low = [spline(n) for n in (5, 4, 3)]
        diff = lambda b: [p - m for p, m in zip(b + [zero], [zero] + b)]  # noqa: E731
        order = [low[0], diff(low[1]), diff(diff(low[2]))]
        ww = [torch.stack(o, -1) * self.per[:, None] ** k for k, o in enumerate(order)]
        out = lambda a, b, c: ww[a][:, 0, :, None, None] * ww[b][:, 1, None, :, None] * ww[c][:, 2, None, None, :]  # noqa: E731
        col = lambda t: t[:, None, None, None]  # noqa: E731
        val = 0 if q is None else col(q) * out(0, 0, 0)
        if mu is not None:
            val = val + col(mu[:, 0]) * out(1, 0, 0) + col(mu[:, 1]) * out(0, 1, 0) + col(mu[:, 2]) * out(0, 0, 1)
        if th is not None:
            t = th / 3
            val = val + col(t[:, 0, 0]) * out(2, 0, 0) + col(t[:, 1, 1]) * out(0, 2, 0) + col(t[:, 2, 2]) * out(0, 0, 2)
            val = val + 2 * (col(t[:, 0, 1]) * out(1, 1, 0) + col(t[:, 0, 2]) * out(1, 0, 1) + col(t[:, 1, 2]) * out(0, 1, 1))
        j = torch.arange(5, device=DEV)
        ix, iy, iz = ((base[:, c, None].long() - j) % self.k[c] for c in range(3))
        at = (ix[:, :, None, None] * self.k[1] + iy[:, None, :, None]) * self.k[2] + iz[:, None, None, :]
        grid = torch.zeros(math.prod(self.k), device=DEV, dtype=F64)
        return grid.index_add(0, at.reshape(-1), val.reshape(-1)).view(self.k)

    def potential(self, grid):
        return torch.fft.ifftn(self.g * torch.fft.fftn(grid)).real


def _own_kernel(r, n):
    return [b - e for b, e in zip(_bare_kernel(r, n), _erfc_kernel(r, n))]


def _per_water(t, which):
    return t[:, which].flatten(0, 1)


def _solve(case, x0, mp, need_forces=True):
    """Energy terms of every molecule pair's share, forces and induced dipoles of the waters at x0."""
    x = x0.clone().requires_grad_(need_forces)
    geo = _geometry(x, mp)
    pts, mu, th = (t.detach().requires_grad_(need_forces) for t in geo)
    q, ke, m = mp[..., 0], P["ke"], x.shape[0]
    pair = _Pairs(x0, case)
    per = pair.periodic
    grid = _Grid(case) if per else None
    both = lambda i, j, sh: ((pts[i], q[i], mu[i], th[i]), (pts[j] + sh, q[j], mu[j], th[j]))  # noqa: E731
    alpha = _vec(*ALPHA)
    grow = [torch.zeros_like(t) for t in (pts, mu, th)]

    def add(e):
        if need_forces:
            for s, g in zip(grow, torch.autograd.grad(e, (pts, mu, th), allow_unused=True)):
                if g is not None:
                    s += g

    def lone_potential(w, src):
        d = w[0][:, 5:, None] - src[0][:, None, :5]
        r = d.norm(dim=-1)
        g = _erfc_kernel(r, 2) if per else _bare_kernel(r, 2)
        phi = _field(d, g, src[2][:, None].expand_as(d), src[3][:, None].expand(*d.shape, 3), src[1][:, None])[0]
        return ke * (phi * (r < pair.rc)).sum(-1)

    def atom_field(w, src):
        """Gradient of the damped potential of src's multipoles at the atoms of w."""
        d = w[0][:, :3, None] - src[0][:, None, :5]
        r = d.norm(dim=-1)
        g = _thole_kernel(r, alpha[:3, None] * alpha, per, 3)
        grad = _field(d, g, src[2][:, None].expand_as(d), src[3][:, None].expand(*d.shape, 3), src[1][:, None])[1]
        return (grad * (r < pair.rc)[..., None]).sum(2)

    def dipole_kernels(xi, xj):
        d = xi[:, :3, None] - xj[:, None, :3]
        r = d.norm(dim=-1)
        g = _thole_kernel(r, alpha[:3, None] * alpha[:3], per, 2)
        inside = (r < pair.rc).to(F64)
        return d, g[1] * inside, g[2] * inside

    # permanent potentials on the lone pairs, fields on the atoms, and the dipole products' pair list
    v, field, held = torch.zeros((m, 2), device=DEV, dtype=F64), torch.zeros((m, 3, 3), device=DEV, dtype=F64), []
    with torch.no_grad():
        for i, j, sh in pair:
            a, b = both(i, j, sh)
            if case["do"] != "dipoles":
                v.index_add_(0, i, lone_potential(a, b)).index_add_(0, j, lone_potential(b, a))
            field.index_add_(0, i, -atom_field(a, b)).index_add_(0, j, -atom_field(b, a))
            held.append((i, j, *dipole_kernels(a[0], b[0])))

    ia, ib = (torch.tensor(k, device=DEV) for k in zip(*[(a, b) for a in range(5) for b in range(a)]))
    fa, fs = (torch.tensor(k, device=DEV) for k in zip(*[(a, b) for a in range(3) for b in range(5) if a != b]))
    la, ls = (torch.tensor(k, device=DEV) for k in zip(*[(a, b) for a in (5, 6) for b in range(5)]))
    pa, pb = (torch.tensor(k, device=DEV) for k in ((1, 2, 2), (0, 0, 1)))
    self_dip = 4 * EW ** 3 / (3 * math.sqrt(math.pi))

    def own(t, s, n):
        d = pts[:, t] - pts[:, s]
        return d, _own_kernel(d.norm(dim=-1), n)

    def permanent_grid():
        return grid.spread(_per_water(pts, range(5)), q.flatten(), mu.flatten(0, 1), th.flatten(0, 1))

    def dipole_linear(d, psi):
        """-d . (reciprocal, self and own-molecule field), over ke on the outside."""
        e = (grid.spread(_per_water(pts, range(3)), None, d.flatten(0, 1), None) * psi).sum()
        dist, g = own(fa, fs, 3)
        grad = _field(dist, g, mu[:, fs], th[:, fs], q[:, fs])[1]
        return e - ke * self_dip * (d * mu[:, :3]).sum() - ke * (d[:, fa] * grad).sum()

    def dipole_quadratic(d):
        """1/2 d T d without the diagonal: reciprocal, self and own-molecule parts."""
        s = grid.spread(_per_water(pts, range(3)), None, d.flatten(0, 1), None)
        dist, g = own(pa, pb, 2)
        own_e = -(_dot(d[:, pa], dist) * _dot(d[:, pb], dist) * g[2] + _dot(d[:, pa], d[:, pb]) * g[1])
        e = 0.5 * (s * grid.potential(s)).sum()
        return e - 0.5 * ke * self_dip * (d * d).sum() - ke * own_e.sum()

    def lone_linear(lam, psi):
        """lam . (reciprocal and own-molecule potential of the lone pairs)."""
        e = (grid.spread(_per_water(pts, range(5, 7)), lam.flatten(), None, None) * psi).sum()
        dist, g = own(la, ls, 2)
        phi = _field(dist, g, mu[:, ls], th[:, ls], q[:, ls])[0]
        return e - ke * (lam[:, la - 5] * phi).sum()

    if per:
        with torch.no_grad():
            psi = grid.potential(permanent_grid())
        with torch.enable_grad():
            z2, z3 = torch.zeros_like(v).requires_grad_(), torch.zeros_like(field).requires_grad_()
            v += torch.autograd.grad(lone_linear(z2, psi), z2)[0].detach()
            field -= torch.autograd.grad(dipole_linear(z3, psi), z3)[0].detach() / ke

    def product(d):
        out = d / alpha[:3, None]
        if per:
            with torch.enable_grad():
                z = d.clone().requires_grad_()
                out = out + torch.autograd.grad(dipole_quadratic(z), z)[0] / ke
        for i, j, r, g1, g2 in held:
            di, dj = d[i][:, :, None], d[j][:, None]
            out.index_add_(0, i, -(g1[..., None] * dj + (g2 * _dot(dj, r))[..., None] * r).sum(2))
            out.index_add_(0, j, -(g1[..., None] * di + (g2 * _dot(di, r))[..., None] * r).sum(1))
        return out

    with torch.no_grad():   # preconditioned conjugate gradient far below the run's tolerance
        dip = alpha[:3, None] * field
        res = field - product(dip)
        z = alpha[:3, None] * res
        p, rz = z, (res * z).sum()
        for _ in range(100):
            if float(z.square().sum(-1).mean().sqrt()) * P["debye"] < 1e-11:
                break
            ap = product(p)
            step = rz / (p * ap).sum()
            dip, res = dip + step * p, res - step * ap
            z = alpha[:3, None] * res
            old, rz = rz, (res * z).sum()
            p = z + rz / old * p
    del held
    if case["do"] == "dipoles":
        return None, None, dip

    def own_potential():
        cols = []
        for a in range(3):
            s = [k for k in range(5) if k != a]
            cols.append(ke * (q[:, s] / (pts[:, a, None] - pts[:, s]).norm(dim=-1)).sum(-1))
        return torch.stack(cols, -1)

    terms = {k: torch.zeros(m, device=DEV, dtype=F64) for k in TERMS[:-1]}   # by the first water of a pair
    lam, kap = torch.zeros_like(v), torch.zeros((m, 3), device=DEV, dtype=F64)
    vint = own_potential().detach()
    for i, j, sh in pair:
        a, b = both(i, j, sh)
        el, pe = _charges_pair(pair, per, a, b)
        di, xd = _dispersion_pair(pair, a, b)
        vl, vi = v.clone().requires_grad_(), vint.clone().requires_grad_()
        ct = _transfer_pair(pair, a, b, vl[i], vi[j]) + _transfer_pair(pair, b, a, vl[j], vi[i])
        re = _repulsion_pair(pair, a, b)
        for k, e in (("elec", el), ("pen", pe), ("rep", re), ("disp", di), ("xdisp", xd), ("ct", ct)):
            terms[k].index_add_(0, i, e.detach())
        if need_forces:
            e = (el + pe + re + di + xd + ct).sum()
            got = torch.autograd.grad(e, (pts, mu, th, vl, vi))
            for s, g in zip(grow + [lam, kap], got):
                s += g
    terms["pol"] -= 0.5 * ke * (dip * field).sum((1, 2))
    more = 0.0
    if per:
        if need_forces:
            e = _recip_energy(grid, permanent_grid(), pts, q, mu, th, own, ia, ib)
            more = float(e.detach())
            add(e)
    if need_forces:
        add((kap * own_potential()).sum())
        for i, j, sh in pair:
            a, b = both(i, j, sh)
            d, g1, g2 = dipole_kernels(a[0], b[0])
            di, dj = dip[i], dip[j]
            e = (lam[i] * lone_potential(a, b)).sum() + (lam[j] * lone_potential(b, a)).sum()
            e = e + ke * ((di * atom_field(a, b)).sum() + (dj * atom_field(b, a)).sum())
            di, dj = di[:, :, None], dj[:, None]
            add(e - ke * (g2 * _dot(di, d) * _dot(dj, d) + g1 * _dot(di, dj)).sum())
        if per:
            psi = grid.potential(permanent_grid())
            add(lone_linear(lam, psi) + dipole_linear(dip, psi) + dipole_quadratic(dip))
        torch.autograd.backward(geo, grow)
    terms["elec"][0] += more
    return terms, -x.grad, dip


def _recip_energy(grid, charge, pts, q, mu, th, own, ia, ib):
    """Reciprocal energy, less the Gaussian self terms and the own-molecule part."""
    e = 0.5 * (charge * grid.potential(charge)).sum()
    s = (q * q).sum() + 2 * EW ** 2 / 3 * (mu * mu).sum() + 8 * EW ** 4 / 45 * (th * th).sum()
    d, g = own(ia, ib, 4)
    phi, grad, second = _field(d, g, mu[:, ib], th[:, ib], q[:, ib], True)
    u = q[:, ia] * phi + _dot(mu[:, ia], grad) + second(th[:, ia]) / 3
    return e - P["ke"] * (EW / math.sqrt(math.pi) * s + u.sum())


def exact(case, seed):
    if case["do"] == "md":
        return None   # a whole trajectory
    x, mp = _inputs(case, seed)
    terms, forces, dip = _solve(case, x, torch.tensor(mp, device=DEV))
    if case["do"] == "dipoles":
        return {"mu": dip.reshape(-1)}
    total = {k: float(t.sum()) for k, t in terms.items()}
    out = {"terms": {**total, "total": sum(total.values())}, "forces": forces.reshape(-1)}
    if case["do"] == "virial":
        out["virial"] = None   # the strain derivative of the whole lattice sum is not formed here
    if case["do"] == "clusters":
        of = torch.repeat_interleave(torch.arange(case["clusters"], device=DEV),
                                     torch.tensor(_sizes(case), device=DEV))
        by = torch.stack([torch.zeros(case["clusters"], device=DEV, dtype=F64).index_add(0, of, terms[k])
                          for k in TERMS[:-1]], -1)
        out["clusters"] = torch.cat([by, by.sum(-1, keepdim=True)], -1)
    return out
