"""Performance cases: whole force computations through the package's public calls.

Every case is one problem dictionary (or a few requests in flight together), planned once and run
to its force and its per-simulation contributions.  Sizes follow the configurations of
`workloads`: the plates cell (60 x 40), the piston sweep (400 x 80..280 cells, resolution 40), the
k_z waveguides (256 x 256 with a 32-cell CPML frame, and the serving mix's smaller cells), the
grooved Bloch membranes (128 x 512), the silicon/silica grating (resolution 40), the cylindrical
piston and the sphere over the notched substrate.  The numbers of time steps, harmonics and
k-points are cut so that a pass takes at most a fraction of a second; a run's steps all cost the
same.  The seed moves the conductivity of the contour and the objects by whole cells or their
permittivities by a few per cent.
"""
import math

import numpy as np
import torch

import workloads as W
from paper_0906_5170_gb300 import Context

# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------


def listed():
    return [
        # the smallest configuration, as a user first runs it: FP64 plates, open line, 24 simulations
        dict(name="plates_fp64", kind="plates", nx=60, ny=40, n_harm=8, steps=4000, precision="fp64"),
        # a coarse piston: the size at which a geometry is set up and tests run
        dict(name="piston_small", kind="piston", nx=60, ny=20, n_harm=6, steps=600, pol="TE+TM", precision="fp32"),
        # one geometry of the piston sweep at its grid (ragged in y), all 640 simulations
        dict(name="piston_sweep", kind="piston", nx=400, ny=166, n_harm=40, steps=1536, pol="TE+TM", precision="fp32"),
        # the serving mix's largest piston grid
        dict(name="piston_512", kind="piston", nx=512, ny=512, n_harm=16, steps=480, pol="TE+TM", precision="fp32"),
        # an odd grid in FP64, as a convergence check of the piston uses
        dict(name="piston_fp64_odd", kind="piston", nx=251, ny=93, n_harm=7, steps=400, pol="TE+TM", precision="fp64"),
        # k_z waveguides at their grid: CPML on four sides, one Lorentz pole, real fields
        dict(name="waveguides_256", kind="waveguide", n=256, n_harm=10, nk=4, steps=480, precision="fp32"),
        # a waveguide request of the serving mix
        dict(name="waveguides_96", kind="waveguide", n=96, n_harm=12, nk=4, steps=720, precision="fp32"),
        # grooved membranes of the serving mix: Bloch k_x, complex fields, CPML along y
        dict(name="grating_bloch", kind="grating", nx=128, ny=512, n_harm=8, nk=4, steps=320, precision="fp32"),
        # silicon guides over silica: three Lorentz poles, complex fields, Bloch k_x and k_z
        dict(name="grating_silica", kind="silica", resolution=40, n_harm=8, nkx=2, nkz=4, steps=240, precision="fp32"),
        # the piston rotated about its axis: (r, z) cells, m = 0, 1, 2
        dict(name="cylinder", kind="cylinder", resolution=40, h=1.0, n_harm=3, mmax=2, steps=1500, precision="fp32"),
        # sphere over the notched substrate in three dimensions with a CPML shell
        dict(name="sphere_cpml", kind="sphere", n=128, pml=12, n_harm=2, steps=80, precision="fp32"),
        # requests of different kinds in flight together, as the serving loop holds them
        dict(name="serving_mix", kind="mix", side=96, steps=480, precision="fp32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds; its steps are cut so that it costs no more than the largest."""
    kind = rng.choice(["plates", "piston", "piston", "piston", "piston", "waveguide", "waveguide", "grating",
                       "silica", "cylinder", "sphere", "mix"])
    if kind == "plates":
        nx, ny = _log(rng, 40, 200), 4 * _log(rng, 8, 40)
        c = dict(kind=kind, nx=nx, ny=ny, n_harm=rng.randint(2, 12), steps=_log(rng, 600, 4000), precision=rng.choice(["fp64", "fp32"]))
    elif kind == "piston":
        prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        c = dict(kind=kind, nx=_log(rng, 60, 512), ny=_log(rng, 20, 512), n_harm=_log(rng, 4, 40), steps=_log(rng, 300, 2000),
                 pol=rng.choice(["TE+TM", "TE+TM", "TM", "TE"]), precision=prec)
    elif kind == "waveguide":
        c = dict(kind=kind, n=16 * rng.randint(4, 16), n_harm=rng.randint(2, 12), nk=rng.randint(1, 8), steps=_log(rng, 200, 800), precision="fp32")
    elif kind == "grating":
        c = dict(kind=kind, nx=_log(rng, 24, 128), ny=_log(rng, 96, 512), n_harm=rng.randint(2, 8), nk=rng.randint(2, 8), steps=_log(rng, 160, 600), precision="fp32")
    elif kind == "silica":
        c = dict(kind=kind, resolution=rng.choice([20, 24, 28, 32, 36, 40]), n_harm=rng.randint(2, 8), nkx=rng.randint(1, 4), nkz=rng.randint(1, 4),
                 steps=_log(rng, 100, 400), precision="fp32")
    elif kind == "cylinder":
        c = dict(kind=kind, resolution=2 * rng.randint(5, 20), h=rng.choice([0.5, 1.0, 1.5, 2.0]), n_harm=rng.randint(1, 4), mmax=rng.randint(0, 2),
                 steps=_log(rng, 400, 2000), precision=rng.choice(["fp32", "fp32", "fp64"]))
    elif kind == "sphere":
        c = dict(kind=kind, n=4 * _log(rng, 12, 32), pml=rng.choice([0, 8, 10, 12]), n_harm=rng.randint(1, 2), steps=_log(rng, 40, 160), precision="fp32")
    else:
        c = dict(kind=kind, side=16 * rng.randint(3, 7), steps=_log(rng, 200, 500), precision="fp32")
    top = max(_cost(x) for x in listed())
    over = _cost(c) / top
    if over > 1.0:
        c["steps"] = max(24, int(c["steps"] / over))
        if _cost(c) > top:
            c["n_harm"] = max(1, int(c["n_harm"] * top / _cost(c)))
    return c


# ---------------------------------------------------------------------------
# Problem dictionaries
# ---------------------------------------------------------------------------


def _plates(c, rng):
    """Two thin plates in a closed box, one open wall-to-wall line midway between them."""
    nx, ny = c["nx"], c["ny"]
    res = ny / 2.0
    p = W.plates_box_2d(res, nx / res, lines=("inner_up",), n_harm=c["n_harm"], polarization="TM", n_steps=c["steps"])
    p["n"] = [nx, ny, 1]
    return p


def _piston(c, rng):
    """Two PEC blocks between PEC side walls, the stress contour one cell around the right block;
    grid lines throughout, so that any nx x ny holds it."""
    nx, ny = c["nx"], c["ny"]
    res = nx / 10.0
    d = 1.0 / res
    bw, bh, gap = max(4, nx // 10), max(4, min(nx // 10, ny // 3)), max(3, nx // 25)
    xr = nx // 2 + gap // 2
    xl = xr - gap - bw - int(rng.integers(0, 3))
    y0 = (ny - bh) // 2 + int(rng.integers(-1, 2))
    p = W._base(2, (nx, ny, 1), res, c["steps"])
    p["objects"] = [{"shape": "box", "lo": [xl * d, y0 * d, 0.0], "hi": [(xl + bw) * d, (y0 + bh) * d, 0.0], "kind": "pec"},
                    {"shape": "box", "lo": [xr * d, y0 * d, 0.0], "hi": [(xr + bw) * d, (y0 + bh) * d, 0.0], "kind": "pec"}]
    p["faces"] = W.box_faces([(xr - 1) * d, (y0 - 1) * d], [(xr + bw + 1) * d, (y0 + bh + 1) * d], 2)
    p.update(n_harm=min(c["n_harm"], bh + 2, bw + 2), polarization=c["pol"], g_variant="zinv")
    return p


def _waveguide(c, rng):
    n = c["n"]
    res = n / 8.0
    gap = 2.0 * int(rng.integers(2, 4)) / 8.0
    mat = W.waveguide_material()
    kp = W.config3_kz_points(gap, n=c["nk"], resolution=res, medium=mat)
    p = W.config3_waveguides(gap, resolution=res, n_cells=n, pml_units=1.0, n_harm=c["n_harm"], n_steps=c["steps"], k_points=kp)
    de = float(rng.uniform(0.95, 1.0))
    for o in p["objects"]:
        o["delta_eps"] *= de
    return p


def _grating(c, rng):
    """A grooved membrane below a slab, period 1 along x, one Bloch k_x per k-point."""
    nx, ny = c["nx"], c["ny"]
    d = 1.0 / nx
    p = W._base(2, (nx, ny, 1), float(nx), c["steps"])
    pc = max(4, ny // 16)
    p["bc"], p["pml_cells"] = ["periodic", "pml", "pec"], [0, pc, 0]
    eps = 11.7 * float(rng.uniform(0.95, 1.05))
    t, gap, mid = max(2, ny // 16), max(4, ny // 12), ny // 2
    yb, yt = mid - gap // 2, mid + (gap + 1) // 2
    box = lambda x0, x1, a, b: {"shape": "box", "lo": [x0, a * d, 0.0], "hi": [x1, b * d, 0.0], "kind": "dielectric", "eps": eps, "mu": 1.0}  # noqa: E731
    p["objects"] = [box(0.0, 1.0, yb - 2 * t, yb - t), box(0.25, 0.75, yb - t, yb), box(0.0, 1.0, yt, yt + t)]
    lo, hi = (yt - 1) * d, (yt + t + 1) * d
    p["faces"] = [{"axis": 1, "sign": -1, "pos": lo, "lo": [0.0, lo, 0.0], "hi": [1.0, lo, 0.0]},
                  {"axis": 1, "sign": 1, "pos": hi, "lo": [0.0, hi, 0.0], "hi": [1.0, hi, 0.0]}]
    p.update(n_harm=min(c["n_harm"], nx), polarization="full", force_axis=1,
             k_points=[{"k": [2 * math.pi * m / c["nk"], 0.0, 0.0], "weight": 1.0 / c["nk"]} for m in range(c["nk"])])
    return p


def _silica(c, rng):
    p = W.grating_silica(0.5, resolution=c["resolution"], nk_x=c["nkx"], nk_z=c["nkz"], n_harm=c["n_harm"], courant=0.2, kz_max=12.0)
    p["n_steps"] = c["steps"]
    return p


def _cylinder(c, rng):
    p = W.cylinder_blocks(c["h"], resolution=c["resolution"], m_list=tuple(range(c["mmax"] + 1)), n_harm=c["n_harm"])
    p["n_steps"] = c["steps"]
    d = int(rng.integers(0, 3)) / c["resolution"]
    p["objects"][0]["lo"][1] -= d
    p["objects"][0]["hi"][1] -= d
    return p


def _sphere(c, rng):
    n = c["n"]
    p = W.config4_sphere_notch(float(rng.uniform(0.3, 0.6)), seed=int(rng.integers(0, 1000)), resolution=n / 4.0, n_cells=n,
                               pml_cells=max(4, c["pml"]), n_harm=c["n_harm"], n_steps=c["steps"])
    if c["pml"] == 0:
        p["bc"], p["pml_cells"] = ["pec", "pec", "pec"], [0, 0, 0]
    return p


def _mix(c):
    s, t = c["side"], c["steps"]
    return [dict(kind="piston", nx=2 * s, ny=s, n_harm=12, steps=t, pol="TE+TM", precision="fp32"),
            dict(kind="waveguide", n=s, n_harm=4, nk=2, steps=t, precision="fp32"),
            dict(kind="piston", nx=s + 3, ny=s - 5, n_harm=8, steps=2 * t, pol="TE+TM", precision="fp32"),
            dict(kind="grating", nx=s // 2, ny=2 * s, n_harm=4, nk=2, steps=t, precision="fp32"),
            dict(kind="sphere", n=s // 2, pml=6, n_harm=1, steps=t // 4, precision="fp32")]


_BUILD = {"plates": _plates, "piston": _piston, "waveguide": _waveguide, "grating": _grating, "silica": _silica,
          "cylinder": _cylinder, "sphere": _sphere}


def _parts(case):
    return _mix(case) if case["kind"] == "mix" else [case]


def _problem(c, seed):
    rng = np.random.default_rng([seed, 17])
    p = _BUILD[c["kind"]](c, rng)
    p["sigma"] = float(rng.uniform(0.9, 1.1))
    p["precision"] = c["precision"]
    return p


# ---------------------------------------------------------------------------
# The passes
# ---------------------------------------------------------------------------

_CTX = []


def _context():
    """The process's context: a program opens one and plans everything on it."""
    if not _CTX:
        _CTX.append(Context(0))
    return _CTX[0]


def prepare(case, seed):
    ctx = _context()
    return [ctx.plan(_problem(c, seed + 1000 * i)) for i, c in enumerate(_parts(case))]


def run(state):
    if len(state) == 1:
        force, per_sim, _ = state[0].run(per_sim=True)
        return {"force": force, "per_sim": per_sim}
    tickets = [plan.submit(tag=i) for i, plan in enumerate(state)]
    return {"forces": [t.force(-1)[0] for t in tickets]}


# ---------------------------------------------------------------------------
# Work: the material ids, weights and results moved once; the arithmetic of the leapfrog
# ---------------------------------------------------------------------------


def _sims_of(p):
    """(k-point, face, harmonics, family, kind, component) of every simulation, in the plan's order:
    a face normal to the force takes every source component, another face its normal's only."""
    fams = {"TM": [("TM", 0, 2), ("TM", 1, 0), ("TM", 1, 1)], "TE": [("TE", 0, 0), ("TE", 0, 1), ("TE", 1, 2)],
            "full": [("full", k, c) for k in (0, 1) for c in range(3)]}
    fam = sum((fams[f] for f in ("TM", "TE") if f in p["polarization"]), []) if p["polarization"] != "full" else fams["full"]
    d = 1.0 / p["resolution"]
    out = []
    for ki in range(len(p["k_points"])):
        for fi, f in enumerate(p["faces"]):
            cnt = [int(round((f["hi"][b] - f["lo"][b]) / d)) for b in range(p["dims"]) if b != f["axis"]]
            nh = [min(p["n_harm"], x) for x in cnt]
            harm = [(a,) for a in range(nh[0])] if len(nh) == 1 else [(a, b) for a in range(nh[0]) for b in range(nh[1])]
            for h in harm:
                out += [(ki, fi, h, fm, kd, c) for fm, kd, c in fam if f["axis"] == p["force_axis"] or c == f["axis"]]
    return out


def _updates(p):
    return float(np.prod(p["n"])) * p["n_steps"] * len(_sims_of(p))


def _flops(p):
    """Arithmetic of one cell-update: differences, products and sums of the leapfrog; slab cells add
    the CPML recursion, dispersive cells their poles; complex fields count twice."""
    N = float(np.prod(p["n"]))
    if p["polarization"] != "full":
        per = 12.0
    else:
        cplx = any(p["bc"][a] == "periodic" and k["k"][a] != 0.0 for a in range(p["dims"]) for k in p["k_points"])
        per = 50.0
        for a in range(p["dims"]):
            if p["bc"][a] == "pml":
                per += 4 * 5.0 * 2 * p["pml_cells"][a] / p["n"][a]
        for o in p["objects"]:
            if o["kind"] == "lorentz":
                vol = np.prod([max(0.0, min(o["hi"][a], p["n"][a] / p["resolution"]) - max(o["lo"][a], 0.0)) for a in range(p["dims"])])
                poles = len(np.atleast_1d(o["omega0"]))
                per += 3 * 8.0 * poles * vol * p["resolution"] ** p["dims"] / N
        per *= 2.0 if cplx else 1.0
    return per * _updates(p)


def work(case):
    b = f = 0.0
    for i, c in enumerate(_parts(case)):
        p = _problem(c, 1000 * i)
        b += float(np.prod(p["n"])) + 8.0 * p["n_steps"] + 16.0 * len(_sims_of(p))
        f += _flops(p)
    return {"bytes": b, "flops": f}


# time per unit of arithmetic relative to the 2D TM/TE runs in FP32
_RATE = {"plates": 1.0, "piston": 1.0, "cylinder": 1.6, "waveguide": 1.2, "grating": 0.9, "silica": 3.5, "sphere": 1.9}


def _cost(c):
    """Relative time of a case: its arithmetic, weighted by the rates of the run kinds."""
    return sum(_flops(_problem(x, 0)) * _RATE[x["kind"]] * (16.0 if x["precision"] == "fp64" else 1.0) for x in _parts(c))


# ---------------------------------------------------------------------------
# The same forces in plain torch with 64-bit arithmetic
# ---------------------------------------------------------------------------

_OFF = {0: ((0.5, 0.0, 0.0), (0.0, 0.5, 0.0), (0.0, 0.0, 0.5)), 1: ((0.0, 0.5, 0.5), (0.5, 0.0, 0.5), (0.5, 0.5, 0.0))}


def _materials(p, grids):
    """eps, mu, PEC and PMC masks and the poles at the points of three broadcastable coordinate arrays."""
    shape = np.broadcast(*grids).shape
    tol = 1e-6 / p["resolution"]
    eps, mu = np.full(shape, p["background"]["eps"]), np.full(shape, p["background"]["mu"])
    pec, pmc = np.zeros(shape, bool), np.zeros(shape, bool)
    de, w0 = np.zeros((3,) + shape), np.zeros((3,) + shape)
    for o in p["objects"]:
        if o["shape"] == "box":
            m = np.ones(shape, bool)
            for a in range(p["dims"]):
                m = m & (grids[a] >= o["lo"][a] - tol) & (grids[a] <= o["hi"][a] + tol)
        else:
            m = np.broadcast_to(sum((grids[a] - o["center"][a]) ** 2 for a in range(p["dims"])) <= (o["radius"] + tol) ** 2, shape)
        pec[m], pmc[m] = o["kind"] == "pec", o["kind"] == "pmc"
        de[:, m] = w0[:, m] = 0.0
        if o["kind"] == "dielectric":
            eps[m], mu[m] = o.get("eps", 1.0), o.get("mu", 1.0)
        elif o["kind"] == "lorentz":
            eps[m], mu[m] = o["eps_inf"], 1.0
            for q, (x, y) in enumerate(zip(np.atleast_1d(o["delta_eps"]), np.atleast_1d(o["omega0"]))):
                de[q][m], w0[q][m] = x, y
    return eps, mu, pec, pmc, de, w0


def _site(p, off):
    d = 1.0 / p["resolution"]
    nx, ny, nz = p["n"]
    return [((np.arange(nx) + off[0]) * d)[None, None, :], ((np.arange(ny) + off[1]) * d)[None, :, None],
            ((np.arange(nz) + off[2]) * d)[:, None, None]]


def _weights(p):
    """w_n = 2 dt Im g(-n dt): the closed form of the z-invariant kernel, or the decaying integral
    (sigma^2/pi) int exp(-sigma t u^2) sqrt(1+u^2) (u^2+1/2) du by the trapezoid rule in u = sinh w."""
    s = p["sigma"]
    dt = p["courant"] / p["resolution"]
    t = dt * np.arange(1, p["n_steps"] + 1)
    if p["g_variant"] == "zinv":
        return 2 * dt * 0.5 * (2 / t**3 + 1.5 * s / t**2 + 0.5 * s * s / t) / (2 * math.pi)
    out = np.empty_like(t)
    for i, x in enumerate(s * t):
        h = min(1 / 64, 0.2 / math.sqrt(x))
        w = np.arange(0.0, math.asinh(math.sqrt(45.0 / x)) + 0.5 + h, h)
        u, ch = np.sinh(w), np.cosh(w)
        f = np.exp(-x * u * u) * ch * ch * (u * u + 0.5)
        out[i] = s * s / math.pi * h * (f.sum() - 0.5 * f[0])
    return 2 * dt * out


def _stencil(p, bloch, pts, off, cyl):
    """Linear interpolation from the sites with offset `off`: (flat site, weight) arrays per point."""
    d = 1.0 / p["resolution"]
    idx, wgt = [np.zeros(len(pts), int)], [np.ones(len(pts), complex)]
    stride = (1, p["n"][0], p["n"][0] * p["n"][1])
    for a in range(p["dims"]):
        u = pts[:, a] / d - off[a]
        i0 = np.floor(u)
        t = u - i0
        up = t > 1 - 1e-9
        i0 = np.where(up, i0 + 1, i0).astype(int)
        t = np.where(up | (t < 1e-9), 0.0, t)
        ni, nw = [], []
        for b, w in zip(idx, wgt):
            for i, f in ((i0, 1 - t), (i0 + 1, t)):
                q = i // p["n"][a]
                ph = np.where(q == 0, 1.0, 0.0) if cyl and a == 0 else bloch[a] ** q
                ni.append(b + (i - q * p["n"][a]) * stride[a])
                nw.append(w * f * ph)
        idx, wgt = ni, nw
    return np.stack(idx, 1), np.stack(wgt, 1)


class _Lattice:
    """Site coefficients of a problem as CUDA tensors, shared by its k-points (their masks on the
    axis of a cylinder apart)."""

    def __init__(self, p, m, dev):
        self.p, self.cyl = p, p.get("coords") == "cylindrical"
        T = lambda x: torch.as_tensor(np.ascontiguousarray(x), device=dev)  # noqa: E731
        tol = 1e-6 / p["resolution"]
        self.ce, self.ch, self.poles = [], [], [[], [], []]
        for c in range(3):
            g = _site(p, _OFF[0][c])
            eps, mu, pec, pmc, de, w0 = _materials(p, g)
            for a in range(p["dims"]):
                if _OFF[0][c][a] == 0.0:
                    wall = np.abs(g[a]) < tol
                    if self.cyl and a == 0:
                        pec = pec | (wall & (c == 2 or m != 0))
                    elif p["bc"][a] != "periodic":
                        pec = pec | wall
            self.ce.append(T(np.where(pec, 0.0, 1 / eps)))
            for q in range(3):
                dq = np.where(pec, 0.0, de[q])
                if dq.any():
                    self.poles[c].append((T(dq), T(w0[q])))
            g = _site(p, _OFF[1][c])
            eps, mu, pec, pmc, _, _ = _materials(p, g)
            if self.cyl and c == 0:
                pmc = pmc | (np.abs(g[0]) < tol)
            self.ch.append(T(np.where(pmc, 0.0, 1 / mu)))
        d, dt = 1 / p["resolution"], p["courant"] / p["resolution"]
        self.d, self.dt, self.pml = d, dt, {}
        for a in range(p["dims"]):
            if p["bc"][a] == "pml":
                for half in (0, 1):
                    n, w = p["n"][a], p["pml_cells"][a] * d
                    x = (np.arange(n) + 0.5 * half) * d
                    rho = np.clip(np.maximum((w - x) / w, (x - (n * d - w)) / w), 0.0, 1.0)
                    sg, al = -4 * math.log(1e-8) / (2 * w) * rho**3, 0.05 * (1 - rho)
                    b = np.exp(-(sg + al) * dt)
                    cc = np.where(sg > 0, sg / np.where(sg > 0, sg + al, 1.0) * (b - 1), 0.0)
                    shape = [1, 1, 1, 1]
                    shape[3 - a] = n
                    self.pml[a, half] = T(b).reshape(shape), T(cc).reshape(shape)


def _march(lat, magnetic, ecomp, hcomp, kz, bloch, mphi, src, meas, gw):
    """Leapfrog of one batch (simulations along dimension 0): src (component -> initial flux), meas
    a list of (rows, component, sites, weights); returns sum_n w_n Re s(n) per simulation."""
    p, d, dt = lat.p, lat.d, lat.dt
    some = next(iter(src.values()))
    dev, S, cx = some.device, some.shape[0], some.dtype
    zero = lambda: torch.zeros((S,) + tuple(reversed(p["n"])), dtype=cx, device=dev)  # noqa: E731
    E, H = {c: zero() for c in ecomp}, {c: zero() for c in hcomp}
    D, B = {c: zero() for c in ecomp}, {c: zero() for c in hcomp}
    P = {(c, q): [zero(), zero()] for c in ecomp for q in range(len(lat.poles[c]))}
    psi = {}
    sg = p["sigma"]
    a_s, b_s = (1 - 0.5 * sg * dt) / (1 + 0.5 * sg * dt), dt / (1 + 0.5 * sg * dt)

    def shifted(F, a, s):
        G = torch.roll(F, -s, 3 - a)
        if bloch is not None and p["bc"][a] == "periodic":
            sl = [slice(None)] * 4
            sl[3 - a] = slice(-1, None) if s > 0 else slice(0, 1)
            G[tuple(sl)] *= bloch[a] if s > 0 else bloch[a].conj()
        return G

    def diff(F, a, s, key):
        """Forward (s = 1) or backward difference along a, stretched inside CPML."""
        if a == 2 and p["dims"] == 2:
            return 1j * kz * F if kz is not None else None
        g = (shifted(F, a, 1) - F) / d if s > 0 else (F - shifted(F, a, -1)) / d
        if a in (0, 1, 2) and (a, 0) in lat.pml:
            b, c = lat.pml[a, 1 if s > 0 else 0]
            psi[key] = b * psi[key] + c * g if key in psi else c * g
            g = g + psi[key]
        return g

    def curl(F, c, s):
        if lat.cyl:
            return curl_cyl(F, c, s)
        a1, a2 = (c + 1) % 3, (c + 2) % 3
        t1 = diff(F[a2], a1, s, (c, a1, s)) if a2 in F else None
        t2 = diff(F[a1], a2, s, (c, a2, s)) if a1 in F else None
        return -t2 if t1 is None else t1 if t2 is None else t1 - t2

    if lat.cyl:
        i = torch.arange(p["n"][0], dtype=torch.float64, device=dev)
        ri, rh, rp, rl = i * d, (i + 0.5) * d, (i + 1) * d, (i - 0.5) * d
        inv = torch.where(i > 0, 1 / torch.where(i > 0, ri, torch.ones_like(ri)), torch.zeros_like(ri))

        def outer(F):
            G = torch.roll(F, -1, 3)
            G[..., -1] = 0
            return G

        def inner(F):
            G = torch.roll(F, 1, 3)
            G[..., 0] = 0
            return G

    def curl_cyl(F, c, s):
        im = 1j * mphi if cx.is_complex else 0.0
        if s > 0:      # curl E at the H sites; components 0, 1, 2 are r, z, phi
            if c == 0:
                return im * inv * F[1] - (shifted(F[2], 1, 1) - F[2]) / d
            if c == 1:
                return (rp * outer(F[2]) - ri * F[2]) / (rh * d) - im / rh * F[0]
            return (shifted(F[0], 1, 1) - F[0]) / d - (outer(F[1]) - F[1]) / d
        if c == 0:
            return im / rh * F[1] - (F[2] - shifted(F[2], 1, -1)) / d
        if c == 1:
            g = (rh * F[2] - rl * inner(F[2])) * inv / d - im * inv * F[0]
            g[..., 0] = 4 * F[2][..., 0] / d
            return g
        return (F[0] - shifted(F[0], 1, -1)) / d - (F[1] - inner(F[1])) / d

    def to_e():
        for c in ecomp:
            t = D[c]
            for q in range(len(lat.poles[c])):
                t = t - P[c, q][0]
            E[c] = t * lat.ce[c]

    def to_h():
        for c in hcomp:
            H[c] = B[c] * lat.ch[c]

    def poles(first):
        for (c, q), st in P.items():
            de, w0 = lat.poles[c][q]
            w2 = (w0 * dt) ** 2
            new = 0.5 * ((2 - w2) * st[0] + de * w2 * E[c]) if first else \
                ((2 - w2) * st[0] - (1 - 0.5 * sg * dt) * st[1] + de * w2 * E[c]) / (1 + 0.5 * sg * dt)
            P[c, q] = [new, st[0]]

    flux = B if magnetic else D
    for c, v in src.items():
        flux[c] += v
    to_h() if magnetic else to_e()
    out = torch.zeros(S, dtype=torch.float64, device=dev)
    for n in range(1, p["n_steps"] + 1):
        h = 0.5 * dt if n == 1 else dt
        if not magnetic:
            for c in hcomp:
                B[c] -= h * curl(E, c, 1)
            to_h()
            poles(n == 1)
            for c in ecomp:
                D[c] = a_s * D[c] + b_s * curl(H, c, -1)
            to_e()
        else:
            poles(False)
            for c in ecomp:
                D[c] += h * curl(H, c, -1)
            to_e()
            for c in hcomp:
                B[c] = a_s * B[c] - b_s * curl(E, c, 1)
            to_h()
        F = H if magnetic else E
        for rows, c, sites, w in meas:
            if c in F:
                v = (F[c][rows].reshape(w.shape[0], -1)[:, sites] * w).sum(1)
                out[rows] += gw[n - 1] * (v.real if v.is_complex() else v)
    return out


def _force(p):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    sims = _sims_of(p)
    d, dims, nx = 1 / p["resolution"], p["dims"], p["n"][0]
    cyl = p.get("coords") == "cylindrical"
    gw = [float(x) for x in _weights(p)]
    N = int(np.prod(p["n"]))
    kps = p["k_points"]
    phases = [[complex(np.exp(1j * k["k"][a] * p["n"][a] * d)) if a < dims and p["bc"][a] == "periodic" else 1.0 + 0j for a in range(3)] for k in kps]
    use_kz = dims == 2 and not cyl and any(k["k"][2] != 0 for k in kps)
    cplx = use_kz or any(ph != 1 for q in phases for ph in q) or any(k.get("m", 0) for k in kps)
    cx = torch.complex128 if cplx else torch.float64
    per = np.zeros(len(sims))
    lats = {}
    # batches: one source kind and family each; a cylinder's lattice depends on m = 0 or not
    keys = sorted({(kd, fm, cyl and kps[ki].get("m", 0) != 0) for ki, _, _, fm, kd, _ in sims})
    for kd, fm, off_axis in keys:
        members = [i for i, s in enumerate(sims) if (s[4], s[3], cyl and kps[s[0]].get("m", 0) != 0) == (kd, fm, off_axis)]
        m_any = kps[sims[members[0]][0]].get("m", 0)
        if off_axis not in lats:
            lats[off_axis] = _Lattice(p, m_any, dev)
        lat = lats[off_axis]
        # simulations whose state fits half of the free memory run together
        size = N * (16 if cplx else 8) * (30 if fm == "full" else 14)
        per_batch = max(1, int((torch.cuda.mem_get_info()[0] if dev.type == "cuda" else 8e9) * 0.5 / size))
        for b0 in range(0, len(members), per_batch):
            rows = members[b0:b0 + per_batch]
            comps = {"TM": ([2], [0, 1]), "TE": ([0, 1], [2]), "full": ([0, 1, 2], [0, 1, 2])}[fm]
            src = {c: torch.zeros((len(rows), N), dtype=cx, device=dev) for c in {sims[i][5] for i in rows}}
            groups = {}
            for r, i in enumerate(rows):
                groups.setdefault((sims[i][0], sims[i][1], sims[i][5]), []).append(r)
            meas = []
            for (ki, fi, c), rs in groups.items():
                f = p["faces"][fi]
                tang = [b for b in range(dims) if b != f["axis"]]
                cnt = [int(round((f["hi"][b] - f["lo"][b]) / d)) for b in tang]
                grid = np.meshgrid(*[np.arange(x) for x in cnt], indexing="ij")
                pts = np.zeros((int(np.prod(cnt)), 3))
                pts[:, f["axis"]] = f["pos"]
                for g, b in zip(grid, tang):
                    pts[:, b] = f["lo"][b] + (g.ravel() + 0.5) * d
                basis = np.ones((len(rs), len(pts)))
                for x, r in enumerate(rs):
                    for n, b, k in zip(sims[rows[r]][2], tang, cnt):
                        L = k * d
                        basis[x] *= math.sqrt(1 / L) if n == 0 else math.sqrt(2 / L) * np.cos(n * math.pi * (pts[:, b] - f["lo"][b]) / L)
                idx, w = _stencil(p, phases[ki], pts, _OFF[kd][c], cyl)
                v = -np.conj(w)[None] * basis[:, :, None] / d
                if cyl:
                    rs_site = (idx % nx + _OFF[kd][c][0]) * d
                    v = v * (pts[:, :1] / np.where(rs_site > 1e-6 * d, rs_site, d / 8))[None]
                put = torch.zeros((len(rs), N), dtype=torch.complex128, device=dev)
                put.index_add_(1, torch.as_tensor(idx.ravel(), device=dev), torch.as_tensor(v.reshape(len(rs), -1), device=dev))
                rt = torch.as_tensor(rs, device=dev)
                src[c][rt] += put if cplx else put.real
                eps, mu = _materials(p, [pts[:, 0], pts[:, 1], pts[:, 2]])[:2]
                base = basis * d ** (dims - 1) * (mu if kd else eps)
                nrm = [0.0] * 3
                nrm[f["axis"]] = float(f["sign"])
                for q, co in ((p["force_axis"], nrm[c]), (c, -0.5 * nrm[p["force_axis"]])):
                    if co:
                        idx, w = _stencil(p, phases[ki], pts, _OFF[kd][q], cyl)
                        ww = (base[:, :, None] * co * w[None]).reshape(len(rs), -1)
                        meas.append((rt, q, torch.as_tensor(idx.ravel(), device=dev), torch.as_tensor(ww if cplx else ww.real.copy(), device=dev)))
            shape = (len(rows),) + tuple(reversed(p["n"]))
            src = {c: v.reshape(shape) for c, v in src.items()}
            col = lambda f: torch.tensor([f(sims[i][0]) for i in rows], dtype=torch.complex128, device=dev).reshape(-1, 1, 1, 1)  # noqa: E731
            bloch = [col(lambda k, a=a: phases[k][a]) for a in range(3)] if cplx and not cyl else None
            kz = col(lambda k: kps[k]["k"][2]) if use_kz else None
            mphi = col(lambda k: kps[k].get("m", 0)) if cplx else 0.0
            per[rows] = _march(lat, kd == 1, comps[0], comps[1], kz, bloch, mphi, src, meas, gw).cpu().numpy()
    per *= np.array([kps[s[0]]["weight"] for s in sims])
    force = np.zeros(3)
    force[p["force_axis"]] = math.fsum(per)
    return force, per


# cell-updates (doubled for complex fields) that the plain form steps through in well under 20 s
_EXACT_MOST = {"plates": 2e10, "piston": 7e10, "waveguide": 1.6e10, "grating": 1e10, "silica": 1e10, "cylinder": 1e10, "sphere": 1.4e10}


def exact(case, seed):
    probs = [(c, _problem(c, seed + 1000 * i)) for i, c in enumerate(_parts(case))]
    if any(_updates(p) > _EXACT_MOST[c["kind"]] for c, p in probs):
        return None
    got = [_force(p) for _, p in probs]
    if torch.cuda.is_available():
        torch.cuda.empty_cache()
    if len(got) == 1:
        return {"force": got[0][0], "per_sim": got[0][1]}
    return {"forces": [f for f, _ in got]}
