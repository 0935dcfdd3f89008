"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is one pass through the public entry points of ``paper_2010_02003_gb300.binding``
with host data in and host data out, as a program that restarts a flood model from a saved
state, advances it to its next output time and keeps the result: ``set_state`` from pinned
memory, ``run_to`` (or single steps), then the state, the gauge series and the mass.  FP32
results are kept in FP32.  ``listed()`` names the standing cases, ``draw()`` gives more of the
same ranges, ``exact()`` states the scheme a second time in plain torch, in 64 bits.

Conditioning: the runs are as long as two programs that differ in rounding only stay together.
In FP64 that is about 100 steps beside wet-dry fronts.  In FP32 it is about 25 steps of the
unlimited scheme beside the channel's banks or for a film around buildings; the limiter's
detector switches beside the banks on the last bit, so limited FP32 runs have no banks.  Runs
start from water that is drawn from the seed, never from a run of this framework.
"""
import math
import random

import numpy as np
import torch

from paper_2010_02003_gb300 import binding as B
from paper_2010_02003_gb300 import inputs

G, TOL, SHOCK = 9.80665, 1e-5, 10.0
CFL_DG2, CFL_FV = 0.33, 0.5
DEFAULTS = {"kind": "run", "scheme": "dg2", "limiter": False, "fp32": False}


def listed():
    return [dict(DEFAULTS, **c) for c in (
        # a small problem stepped by a caller that sets the step size itself (coupling to
        # another model): launches and their gaps are all of it
        {"name": "steps_ll_fp64", "kind": "steps", "site": "basin", "nx": 96, "ny": 80,
         "limiter": True, "steps": 16},
        # the closed 128 x 128 basin with a circular dam, run to 10 s
        {"name": "basin_nl_fp64", "site": "basin", "nx": 128, "ny": 128, "seconds": 10.0},
        # the 2000 x 1000, 2 m floodplain, mostly dry, limited: the repository's headline
        {"name": "floodplain_ll_fp64", "site": "floodplain", "nx": 2000, "ny": 1000, "wet": 0.04,
         "limiter": True, "seconds": 10.0},
        # a ragged floodplain window, unlimited, with more of it under water
        {"name": "floodplain_nl_fp64", "site": "floodplain", "nx": 1237, "ny": 731, "wet": 0.12,
         "seconds": 10.0},
        # the floodplain in FP32 at the height of a flood, for many runs at a survey's accuracy
        {"name": "floodplain_nl_fp32", "site": "floodplain", "nx": 2000, "ny": 1000, "wet": 0.2,
         "fp32": True, "seconds": 2.0},
        # every cell wet (a reservoir, an estuary at high water): the dense rates
        {"name": "flooded_ll_fp64", "site": "flooded", "nx": 1000, "ny": 600, "limiter": True,
         "seconds": 3.0},
        {"name": "flooded_nl_fp32", "site": "flooded", "nx": 2000, "ny": 1000, "fp32": True,
         "seconds": 10.0},
        {"name": "flooded_ll_fp32", "site": "flooded", "nx": 1451, "ny": 1013, "limiter": True,
         "fp32": True, "seconds": 6.0},
        # rain on a city at half a metre: the largest grids, thin films around buildings
        {"name": "urban_nl_fp32", "site": "urban", "nx": 2900, "ny": 2900, "fp32": True,
         "seconds": 1.0},
        # scenarios of uneven sizes advanced together, each with its own step
        {"name": "ensemble_nl_fp32", "kind": "ensemble", "members": 24, "nx": 1024, "ny": 512,
         "fp32": True, "seconds": 4.0},
        # calibration: the misfit's gradient for the Manning field and the inflow
        {"name": "adjoint_fp64", "kind": "adjoint", "nx": 512, "ny": 512, "steps": 40, "slots": 8},
        # the paper's comparator at the same resolution
        {"name": "floodplain_fv2_fp64", "site": "floodplain", "scheme": "fv2", "nx": 2000,
         "ny": 1000, "wet": 0.04, "seconds": 14.0},
    )]


def draw(rng):
    """One more case of the listed ranges."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["basin", "floodplain", "floodplain", "flooded", "flooded", "urban",
                       "ensemble", "adjoint", "fv", "steps"])
    limiter, fp32 = rng.random() < 0.5, rng.random() < 0.5
    if kind == "steps":
        c = {"kind": "steps", "site": "basin", "nx": size(40, 128), "ny": size(40, 128),
             "limiter": limiter, "steps": rng.randint(8, 24)}
    elif kind == "basin":
        c = {"site": "basin", "nx": size(64, 512), "ny": size(64, 512), "limiter": limiter,
             "seconds": round(rng.uniform(3.0, 8.0), 2)}
    elif kind == "floodplain":
        c = {"site": kind, "nx": size(128, 2000), "ny": size(96, 1000),
             "limiter": limiter and not fp32, "fp32": fp32,
             "wet": round(math.exp(rng.uniform(math.log(0.02), math.log(0.4))), 3),
             "seconds": round(rng.uniform(1.0, 2.0) if fp32 else rng.uniform(4.0, 10.0), 2)}
    elif kind == "flooded":
        c = {"site": kind, "nx": size(128, 2000 if fp32 else 1000), "limiter": limiter,
             "ny": size(96, 1000 if fp32 else 600), "fp32": fp32,
             "seconds": round(rng.uniform(1.5, 8.0 if fp32 else 3.0), 2)}
    elif kind == "urban":
        c = {"site": kind, "nx": size(256, 2900), "ny": size(256, 2900), "fp32": True,
             "limiter": limiter,
             "seconds": round(rng.uniform(0.4, 1.0), 2)}
    elif kind == "ensemble":
        c = {"kind": kind, "members": rng.randint(3, 24), "nx": size(256, 1024),
             "ny": size(128, 512), "fp32": True, "seconds": round(rng.uniform(1.5, 4.0), 2)}
    elif kind == "adjoint":
        c = {"kind": kind, "nx": size(64, 512), "ny": size(64, 512), "steps": rng.randint(12, 40),
             "slots": rng.randint(3, 16), "fp32": fp32}
    else:
        c = {"site": "floodplain", "scheme": rng.choice(["fv1", "fv2"]), "nx": size(128, 2000),
             "ny": size(96, 1000), "wet": round(rng.uniform(0.02, 0.4), 3),
             "seconds": round(rng.uniform(4.0, 14.0), 2)}
    return dict(DEFAULTS, **c)


# ---- inputs --------------------------------------------------------------------------------

def modes(f):
    """Average, x-slope and y-slope of a field at the corner nodes (Eq. 3 on face averages)."""
    e, w = 0.5 * (f[:-1, 1:] + f[1:, 1:]), 0.5 * (f[:-1, :-1] + f[1:, :-1])
    n, s = 0.5 * (f[1:, :-1] + f[1:, 1:]), 0.5 * (f[:-1, :-1] + f[:-1, 1:])
    return 0.5 * (e + w), 0.5 * (e - w), 0.5 * (n - s)


def water(site, seed, averages_only=False):
    """The nine planes of the site's initial water, set in a slow seeded motion where it is
    deep enough to carry one."""
    u = np.zeros((9, site.ny, site.nx))
    if site.eta_corner is None:
        return u
    h0, h1x, h1y = modes(site.eta_corner - site.z_corner)
    wet = h0 > 0.0
    u[0], u[1], u[2] = np.where(wet, h0, 0.0), np.where(wet, h1x, 0.0), np.where(wet, h1y, 0.0)
    rng = np.random.Generator(np.random.PCG64(seed + 17))
    a, b = rng.uniform(0.0, 2.0 * np.pi, size=2)
    y, x = np.mgrid[0:site.ny, 0:site.nx]
    deep = u[0] - np.maximum(np.abs(u[1]), np.abs(u[2])) > 0.05
    u[3] = np.where(deep, u[0] * (0.2 + 0.1 * np.sin(2.0 * np.pi * y / 97.0 + a)), 0.0)
    u[6] = np.where(deep, u[0] * 0.1 * np.sin(2.0 * np.pi * x / 131.0 + b), 0.0)
    if averages_only:
        for k in (1, 2, 4, 5, 7, 8):
            u[k] = 0.0
    return u


def flood(nx, ny, seed, wet):
    """The floodplain at the rising limb of its hydrograph: the lowest `wet` of it, the reaches of
    the channel among them, under a free surface that falls slightly eastwards."""
    c = inputs.floodplain(nx=nx, ny=ny, seed=seed, sample_every=1.0)
    x = np.arange(nx + 1) * c.dx
    c.eta_corner = (np.quantile(c.z_corner, wet) + 1e-4 * (0.5 * nx * c.dx - x)[None, :]
                    + np.zeros_like(c.z_corner))
    return c


def high_water(nx, ny, seed):
    c = inputs.flooded_plain(nx=nx, ny=ny, seed=seed,
                             freeboard=random.Random(seed).uniform(0.4, 0.6))
    c.sample_every = 1.0
    return c


def city(nx, ny, seed):
    """Some minutes into the rain: a film over the streets and roofs."""
    c = inputs.urban(nx=nx, ny=ny, seed=seed, nblocks=max(1, int(2000 * nx * ny / 8192.0 ** 2)))
    film = 0.004 + 0.003 * inputs.fbm(ny + 1, nx + 1, 0.8, 1.0, seed + 5)
    c.eta_corner = c.z_corner + film
    c.gauges, c.sample_every = np.array([[0.1 * nx, 0.1 * ny], [0.3 * nx, 0.2 * ny]]), 0.5
    return c


def site_of(case, seed):
    """(the site as an inputs.Case, the time its run starts at)."""
    nx, ny = case["nx"], case["ny"]
    r = random.Random(seed)
    if case["site"] == "basin":
        c = inputs.hump(nx=nx, ny=ny, eta=0.5, dam_eta=r.uniform(0.9, 1.1),
                        dam_radius=20.0 * min(nx, ny) / 128.0, amp=r.uniform(0.75, 0.85),
                        width2=200.0 * (min(nx, ny) / 128.0) ** 2)
        c.gauges, c.sample_every = np.array([[0.25 * nx, 0.25 * ny], [0.75 * nx, 0.5 * ny]]), 0.5
        return c, 0.0
    if case["site"] == "floodplain":
        return flood(nx, ny, seed, case["wet"]), 1800.0
    return (high_water(nx, ny, seed), 1800.0) if case["site"] == "flooded" else (city(nx, ny, seed), 300.0)


def members_of(case, seed):
    """Sites of an ensemble, sizes log-uniform up to nx x ny: rivers at high water with inflows
    and roughness of their own, under rain in every other one."""
    got = []
    for s in range(case["members"]):
        r = random.Random(s)  # the sizes are the case's, the rest is the seed's
        nx = int(round(math.exp(r.uniform(math.log(64), math.log(case["nx"])))))
        ny = int(round(math.exp(r.uniform(math.log(64), math.log(case["ny"])))))
        r = random.Random(1000 * seed + s)
        c = high_water(nx, ny, seed + s)
        c.manning, c.n_uniform = None, r.uniform(0.02, 0.08)
        c.inflows[0].q_knots = c.inflows[0].q_knots * r.uniform(0.25, 2.0)
        c.gauges = c.gauges[::2]
        if s % 2:
            c.rain = (r.uniform(20.0, 80.0) / 3.6e6, 0.0, 1800.0)
        got.append(c)
    return got


def calibration(case, seed):
    """The calibration problem: site, step sizes, sample counts, observed depths, Manning field."""
    c = inputs.flooded_plain(nx=case["nx"], ny=case["ny"], seed=seed)
    rng = np.random.Generator(np.random.PCG64(seed + 3))
    c.manning = rng.uniform(0.03, 0.05, size=(c.ny, c.nx))
    f = c.inflows[0]
    f.t_knots = np.linspace(0.0, 8.0, 64)
    f.q_knots = 15.0 + 5.0 * rng.random(64)
    k = case["steps"]
    dts = np.full(k, 0.08) + 0.01 * rng.random(k)
    samples = list(range(5, k + 1, 5))
    h0, h1x, h1y = modes(c.eta_corner - c.z_corner)
    at = [(min(int(x / c.dx), c.nx - 1), min(int(y / c.dy), c.ny - 1)) for x, y in c.gauges]
    obs = np.array([[h0[j, i] for i, j in at]] * len(samples))
    return c, dts, samples, obs + 0.05 * rng.standard_normal(obs.shape), c.manning, f.q_knots


def pinned(a):
    t = torch.empty(a.shape, dtype=torch.float64, pin_memory=torch.cuda.is_available())
    t.numpy()[...] = a
    return t.numpy()


class Held:
    """One solver with the saved state that it restarts from and the buffers of its results."""

    def __init__(self, case, site, t0, seed, scheme="dg2"):
        kw = {} if scheme == "dg2" else {
            "scheme": {"fv1": B.DG2_SCHEME_FV1, "fv2": B.DG2_SCHEME_FV2}[scheme], "cfl": CFL_FV}
        self.solver = B.solver_from_case(site, variant=B.DG2_LL if case["limiter"] else B.DG2_NL,
                                         precision=B.DG2_FP32 if case["fp32"] else B.DG2_FP64, **kw)
        self.t0, self.fp32, self.site = t0, case["fp32"], site
        self.start = pinned(water(site, seed, scheme != "dg2"))
        self.out = pinned(np.zeros_like(self.start))
        self.kept = torch.empty(self.out.shape, dtype=torch.float32) if self.fp32 else None

    def restart(self):
        self.solver.set_state(self.start, self.t0)

    def results(self):
        B.dg2_get_state(self.solver.ctx, self.site.nx, self.site.ny, out=self.out)
        depths = self.solver.read_gauges(cap=256)[1]
        if self.fp32:
            return {"state": self.kept.copy_(torch.from_numpy(self.out)),
                    "gauges": depths.astype(np.float32)}
        return {"state": self.out, "gauges": depths, "mass": np.array(self.solver.mass())}


def prepare(case, seed):
    if case["kind"] == "adjoint":
        site, dts, samples, obs, man, q = calibration(case, seed)
        adj = B.Adjoint(site, nsnap=case["slots"], max_steps=case["steps"],
                        precision=B.DG2_FP32 if case["fp32"] else B.DG2_FP64)
        adj.set_schedule(dts, samples, obs)
        return {"case": case, "adj": adj, "man": man, "q": q}
    if case["kind"] == "ensemble":
        held = [Held(case, c, 600.0, seed + s) for s, c in enumerate(members_of(case, seed))]
        ens = B.Ensemble([h.solver for h in held])
        ens.set_tile_shape(16, 8)
        return {"case": case, "held": held, "ens": ens}
    site, t0 = site_of(case, seed)
    held = Held(case, site, t0, seed, case["scheme"])
    return {"case": case, "held": held, "dt": 0.02 + 0.01 * random.Random(seed).random()}


def run(state):
    case = state["case"]
    if case["kind"] == "adjoint":
        state["adj"].set_params(state["man"], state["q"])
        loss, by_manning, by_knot = state["adj"].gradient()
        got = {"loss": np.array([loss]), "by_manning": by_manning, "by_knot": by_knot}
        return {k: v.astype(np.float32) for k, v in got.items()} if case["fp32"] else got
    if case["kind"] == "ensemble":
        for h in state["held"]:
            h.restart()
        state["ens"].run_to(600.0 + case["seconds"])
        return [h.results() for h in state["held"]]
    h = state["held"]
    h.restart()
    if case["kind"] == "steps":
        for _ in range(case["steps"]):
            h.solver.step(state["dt"])
    else:
        h.solver.run_to(h.t0 + case["seconds"])
    return h.results()


def work(case):
    """What a pass cannot do without: the state in and out over the host boundary, and for each
    step every computed cell's state read and written once with its bed and Manning n (FP64: 22
    values, FP32: 23), at the scheme's operations per wet cell and step (friction and two stages)."""
    cells, b = case["nx"] * case["ny"], 4 if case["fp32"] else 8
    if case["kind"] == "adjoint":
        # forward once, reverse once (state, adjoint and gradient in and out)
        return {"bytes": case["steps"] * cells * b * (22 + 33), "flops": case["steps"] * cells * 934 * 4}
    wet = 1.0
    if case["kind"] == "ensemble":
        # sizes log-uniform from 64: their mean
        mean = [(n - 64) / math.log(n / 64) for n in (case["nx"], case["ny"])]
        cells, dt = case["members"] * mean[0] * mean[1], 0.09
    elif case["kind"] == "steps":
        dt = None
    else:
        dt = {"basin": 0.075, "floodplain": 0.12, "flooded": 0.09, "urban": 0.05}[case["site"]]
        wet = case.get("wet", 1.0)
    n = case["steps"] if dt is None else case["seconds"] / dt
    per = 934 + (166 if case["limiter"] else 0)
    values = 23 if case["fp32"] else 22
    if case["scheme"] != "dg2":
        n, per, values = n * CFL_DG2 / CFL_FV, 380 if case["scheme"] == "fv2" else 170, 8
    return {"bytes": cells * 144 + n * cells * wet * values * b, "flops": n * cells * wet * per}


# ---- the scheme once more, in plain torch and 64 bits ---------------------------------------

EAST, WEST, NORTH, SOUTH = 0, 1, 2, 3
R3 = math.sqrt(3.0)


def root(x):
    """sqrt with derivative 0 at 0."""
    ok = x > 0.0
    return torch.where(ok, torch.sqrt(torch.where(ok, x, torch.ones_like(x))), torch.zeros_like(x))


def pos(x):
    return torch.where(x > 0.0, x, torch.zeros_like(x))


def larger(a, b):
    return torch.where(a > b, a, b)


def smaller(a, b):
    return torch.where(a < b, a, b)


def speeds(h, qx, qy):
    ok = h > TOL
    d = torch.where(ok, h, torch.ones_like(h))
    return torch.where(ok, qx / d, torch.zeros_like(h)), torch.where(ok, qy / d, torch.zeros_like(h))


def flux(h, qn, qt):
    """Physical flux normal to a face (h, normal and tangential discharge)."""
    u, v = speeds(h, qn, qt)
    return h * u, h * u * u + 0.5 * G * h * h, h * u * v


def hll(a, b):
    """HLL flux between the lower side a and the upper side b, each (h, qn, qt)."""
    da, db = a[0] <= TOL, b[0] <= TOL
    ua, _ = speeds(*a)
    ub, _ = speeds(*b)
    ca, cb = root(G * a[0]), root(G * b[0])
    us, cs = 0.5 * (ua + ub) + ca - cb, 0.5 * (ca + cb) + 0.25 * (ua - ub)
    sl = torch.where(da, ub - 2.0 * cb, torch.where(db, ua - ca, smaller(ua - ca, us - cs)))
    sr = torch.where(da, ub + cb, torch.where(db, ua + 2.0 * ca, larger(ub + cb, us + cs)))
    fa, fb = flux(*a), flux(*b)
    dry = da & db
    left, right = sl >= 0.0, sr <= 0.0
    den = torch.where(dry | left | right, torch.ones_like(sl), sr - sl)
    got = []
    for k in range(3):
        m = (sr * fa[k] - sl * fb[k] + sl * sr * (b[k] - a[k])) / den
        f = torch.where(left, fa[k], torch.where(right, fb[k], m))
        got.append(torch.where(dry, torch.zeros_like(f), f))
    return got


def minmod(a, b, c):
    up, down = (a > 0) & (b > 0) & (c > 0), (a < 0) & (b < 0) & (c < 0)
    zero = torch.zeros_like(a)
    return torch.where(up, smaller(smaller(a, b), c), torch.where(down, larger(larger(a, b), c), zero))


class Plain:
    """The scheme over whole planes: DG2 (with or without local limiting), MUSCL-FV2 or FV1."""

    def __init__(self, site, scheme="dg2", limiter=False, cfl=None):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.put = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
        self.site, self.scheme, self.limiter = site, scheme, limiter
        self.cfl = (CFL_FV if scheme != "dg2" else site.cfl) if cfl is None else cfl
        self.nx, self.ny, self.dx, self.dy = site.nx, site.ny, site.dx, site.dy
        self.z = self.put(np.stack(modes(site.z_corner)))
        man = site.manning if site.manning is not None else np.full((site.ny, site.nx), site.n_uniform)
        self.n = self.put(man)
        f = site.inflows[0] if site.inflows else None
        self.inflow = None
        if f is not None:  # the sites here have inflows on the west edge only
            s = (np.arange(self.ny) + 0.5) * self.dy
            face = (s >= f.s0) & (s <= f.s0 + f.length)
            self.inflow = (self.put(face) > 0, face.sum() * self.dy, f.t_knots, self.put(f.q_knots))

    # boundaries: (h, qx, qy) outside an edge from the cell's own limit
    def ghost(self, edge, lim, t):
        h, qx, qy = lim
        x = edge in (EAST, WEST)
        if self.site.bc[{WEST: 0, EAST: 1, SOUTH: 2, NORTH: 3}[edge]] == inputs.OPEN:
            into = {WEST: qx > 0, EAST: qx < 0, SOUTH: qy > 0, NORTH: qy < 0}[edge]
            got = [h, torch.where(into, 0.0 * qx, qx) if x else qx, qy if x else torch.where(into, 0.0 * qy, qy)]
        else:
            got = [h, -qx if x else qx, qy if x else -qy]
        if edge == WEST and self.inflow is not None:
            face, width, tk, qk = self.inflow
            k = min(max(int(np.searchsorted(tk, t, side="left")), 1), len(tk) - 1)
            w = min(max((t - tk[k - 1]) / (tk[k] - tk[k - 1]), 0.0), 1.0)
            q = (qk[k - 1] + w * (qk[k] - qk[k - 1])) / width
            deep = larger(pos(h), (q * q / G) ** (1.0 / 3.0) + 0.0 * h)
            got = [torch.where(face, deep, got[0]), torch.where(face, q + 0.0 * qx, got[1]),
                   torch.where(face, 0.0 * qy, got[2])]
        return got

    def edge_of(self, a, edge):
        return {EAST: a[:, -1:], WEST: a[:, :1], NORTH: a[-1:], SOUTH: a[:1]}[edge]

    def sides(self, own, out):
        """Lower and upper sides of the x faces and of the y faces from the four own records (per
        field: east, west, north, south) and the four records beyond the edges."""
        xa = [torch.cat([out[WEST][k], own[EAST][k]], 1) for k in range(len(own[EAST]))]
        xb = [torch.cat([own[WEST][k], out[EAST][k]], 1) for k in range(len(own[EAST]))]
        ya = [torch.cat([out[SOUTH][k], own[NORTH][k]], 0) for k in range(len(own[EAST]))]
        yb = [torch.cat([own[SOUTH][k], out[NORTH][k]], 0) for k in range(len(own[EAST]))]
        return (xa, xb), (ya, yb)

    def beyond(self, edge, lim, t):
        """Ghost limit outside an edge, from the cells' own limits there."""
        own = [self.edge_of(a, edge) for a in lim]
        if edge in (EAST, WEST):
            return [a[:, None] for a in self.ghost(edge, [a[:, 0] for a in own], t)]
        return [a[None, :] for a in self.ghost(edge, [a[0] for a in own], t)]

    def face_fluxes(self, x, y):
        """Fluxes of the revised x and y faces as (mass, x-momentum, y-momentum)."""
        fx = hll(*[(h, h * u, h * v) for h, u, v in x])
        g = hll(*[(h, h * v, h * u) for h, u, v in y])
        return fx, [g[0], g[2], g[1]]

    def sources(self, t):
        rain, r0, r1 = self.site.rain
        s = torch.zeros_like(self.n) + (rain if r0 <= t < r1 else 0.0)
        px, py, qp = self.site.point
        if qp != 0.0:
            i, j = min(int(px / self.dx), self.nx - 1), min(int(py / self.dy), self.ny - 1)
            s[j, i] += qp / (self.dx * self.dy)
        return s

    def operator(self, u, t):
        """The nine operator planes of Eqs. 4-5."""
        tol = TOL
        sg = {EAST: (1, 1.0), WEST: (1, -1.0), NORTH: (2, 1.0), SOUTH: (2, -1.0)}
        lim = {f: [u[3 * v] + s * u[3 * v + m] for v in range(3)] for f, (m, s) in sg.items()}
        zf = {f: self.z[0] + s * self.z[m] for f, (m, s) in sg.items()}
        h0 = u[0]
        total = sum(pos(lim[f][0]) for f in sg)
        negative = (lim[0][0] < 0) | (lim[1][0] < 0) | (lim[2][0] < 0) | (lim[3][0] < 0)
        part = (h0 > tol) & negative
        scale = torch.where(part, h0 / torch.where(part, 0.25 * total, torch.ones_like(h0)), torch.ones_like(h0))
        own, out = {}, {}
        for f in sg:
            h, qx, qy = lim[f]
            eps = 0.1 * h0
            thin = (eps > tol) & (h < eps)
            den = torch.where(thin, h * h + eps * eps, torch.ones_like(h))
            a, b = speeds(h, qx, qy)
            a, b = torch.where(thin, 2.0 * pos(h) * qx / den, a), torch.where(thin, 2.0 * pos(h) * qy / den, b)
            hs = torch.where(part, scale * pos(h), pos(h))
            eta = torch.where(part, h + zf[f], zf[f] + pos(h))
            zo = torch.where(part, eta - hs, zf[f])
            own[f] = [h, hs, zo, eta, a, b, part]
            g = self.beyond(f, lim[f], t)
            ga, gb = speeds(*g)
            ze = self.edge_of(zf[f], f)
            out[f] = [g[0], pos(g[0]), ze, ze + pos(g[0]), ga, gb, torch.zeros_like(ze) > 0]
        rev = []
        for a, b in self.sides(own, out):
            mixed = a[6] | b[6]
            zs = larger(a[2], b[2])
            one = []
            for r in (a, b):
                h = torch.where(mixed, pos(r[3] - zs), r[1])
                zz = torch.where(mixed, zs - pos(zs - r[3]), r[2] - pos(-r[0]))
                one.append((h, r[4], r[5], zz))
            rev.append(one)
        (xa, xb), (ya, yb) = rev
        fx, gy = self.face_fluxes([s[:3] for s in (xa, xb)], [s[:3] for s in (ya, yb)])
        dx, dy = self.dx, self.dy
        new = [None] * 9
        for d, (lo, up, fl, dd) in enumerate(((xb, xa, fx, dx), (yb, ya, gy, dy))):
            low = (lambda a: a[:, :-1]) if d == 0 else (lambda a: a[:-1])     # the cell's west / south face
            high = (lambda a: a[:, 1:]) if d == 0 else (lambda a: a[1:])      # its east / north face
            w = [low(lo[0]), low(lo[0]) * low(lo[1]), low(lo[0]) * low(lo[2])]
            e = [high(up[0]), high(up[0]) * high(up[1]), high(up[0]) * high(up[2])]
            z1 = 0.5 * (high(up[3]) - low(lo[3]))
            c0, c1 = [0.5 * (p + q) for p, q in zip(e, w)], [0.5 * (p - q) for p, q in zip(e, w)]
            pts = [[p + s * q / R3 for p, q in zip(c0, c1)] for s in (1.0, -1.0)]
            if d == 0:
                ph = [flux(*p) for p in pts]
            else:
                ph = [(f[0], f[2], f[1]) for f in (flux(p[0], p[2], p[1]) for p in pts)]
            for v in range(3):
                hi, lw = high(fl[v]), low(fl[v])
                l0 = -(hi - lw) / dd
                l1 = (hi + lw) - (ph[0][v] + ph[1][v])
                if v == d + 1:
                    l0 = l0 - 2.0 * G * c0[0] * z1 / dd
                    l1 = l1 + (2.0 * G / 3.0) * c1[0] * z1
                new[3 * v] = l0 if d == 0 else new[3 * v] + l0
                new[3 * v + d + 1] = -(3.0 / dd) * l1
        new[0] = new[0] + self.sources(t)
        return torch.stack(new)

    def friction(self, u, dt):
        def point(h, qx, qy):
            ok = h > TOL
            hh = torch.where(ok, h, torch.ones_like(h))
            d = 1.0 + dt * G * self.n * self.n * root(qx * qx + qy * qy) / (hh * hh * hh ** (1.0 / 3.0))
            return torch.where(ok, qx / d, qx), torch.where(ok, qy / d, qy)

        new = [u[k] for k in range(9)]
        new[3], new[6] = point(u[0], u[3], u[6])
        if self.scheme == "dg2":
            for m in (1, 2):
                p = point(*[u[3 * v] + u[3 * v + m] / R3 for v in range(3)])
                q = point(*[u[3 * v] - u[3 * v + m] / R3 for v in range(3)])
                new[3 + m], new[6 + m] = 0.5 * R3 * (p[0] - q[0]), 0.5 * R3 * (p[1] - q[1])
        return torch.stack(new)

    def limited(self, u):
        new = u.clone()
        for m, ax, h in ((1, 1, self.dx), (2, 0, self.dy)):
            n = u.shape[ax + 1]
            if n < 3:
                continue
            at = lambda a, k: a.narrow(a.dim() - 2 + ax, k, n - 2)  # noqa: E731
            h0 = u[0]
            wet = (at(h0, 0) > TOL) & (at(h0, 1) > TOL) & (at(h0, 2) > TOL)
            for v in range(3):
                k0, k1 = (u[0] + self.z[0], u[m] + self.z[m]) if v == 0 else (u[3 * v], u[3 * v + m])
                c0, c1 = at(k0, 1), at(k1, 1)
                up = ((at(k0, 2) - at(k1, 2)) - (c0 + c1)).abs()
                lo = ((c0 - c1) - (at(k0, 0) + at(k1, 0))).abs()
                size = torch.maximum((c0 - c1 / R3).abs(), (c0 + c1 / R3).abs()).clamp(min=TOL)
                shock = wet & (torch.maximum(up, lo) > SHOCK * (0.5 * h * size))
                s = minmod(c1, at(k0, 2) - c0, c0 - at(k0, 0))
                if v == 0:
                    shock = shock & (s != c1)
                    s = s - at(self.z[m], 1)
                at(new[3 * v + m], 1).copy_(torch.where(shock, s, at(u[3 * v + m], 1)))
        return new

    def dried(self, u):
        """The treatment of dry cells and of fronts after a stage."""
        wet = u[0] > TOL
        eta = u[0] + self.z[0]
        keep = {0: wet}
        for m in (1, 2):
            front = torch.zeros_like(wet)
            for s in (1.0, -1.0):
                front = front | ((u[0] + s * u[m] <= TOL) & ~(self.z[0] + s * self.z[m] > eta))
            keep[m] = wet & ~front
        zero = torch.zeros_like(u[0])
        return torch.stack([u[0]] + [torch.where(keep[k % 3], u[k], zero) for k in range(1, 9)])

    def dg2_step(self, u, t, dt):
        u = self.friction(u, dt)
        if self.limiter:
            u = self.limited(u)
        v = self.dried(u + dt * self.operator(u, t))
        if self.limiter:
            v = self.limited(v)
        return self.dried(0.5 * (u + v + dt * self.operator(v, t + dt)))

    def fv_operator(self, u, t):
        h0, qx, qy = u[0], u[3], u[6]
        own, out = {}, {}
        for ax, (lo, up) in ((1, (WEST, EAST)), (0, (SOUTH, NORTH))):
            n = h0.shape[ax]
            fields = [h0 + self.z[0], h0, qx, qy]
            own[lo], own[up] = [], []
            at = lambda a, k: a.narrow(ax, k, n - 2)  # noqa: E731
            for k in fields:
                s = torch.zeros_like(k)
                if self.scheme == "fv2" and n > 2:
                    wet = (at(h0, 0) > TOL) & (at(h0, 1) > TOL) & (at(h0, 2) > TOL)
                    db, df = at(k, 1) - at(k, 0), at(k, 2) - at(k, 1)
                    ok = wet & (db != 0.0)
                    r = df / torch.where(ok, db, torch.ones_like(db))
                    phi = torch.maximum((1.25 * r).clamp(max=1.0), r.clamp(max=1.25)).clamp(min=0.0)
                    at(s, 1).copy_(torch.where(ok, phi * db, torch.zeros_like(db)))
                own[lo].append(k - 0.5 * s)
                own[up].append(k + 0.5 * s)
        for f in own:
            e = [self.edge_of(a, f) for a in own[f]]
            g = self.beyond(f, own[f][1:], t)
            out[f] = [g[0] + (e[0] - e[1])] + g
        rev = []
        for a, b in self.sides(own, out):
            zs = larger(a[0] - a[1], b[0] - b[1])
            rev.append([(pos(r[0] - zs), *speeds(r[1], r[2], r[3]), zs - pos(zs - r[0])) for r in (a, b)])
        (xa, xb), (ya, yb) = rev
        fx, gy = self.face_fluxes([s[:3] for s in (xa, xb)], [s[:3] for s in (ya, yb)])
        new = torch.zeros_like(u)
        for v in range(3):
            new[3 * v] = -(fx[v][:, 1:] - fx[v][:, :-1]) / self.dx - (gy[v][1:] - gy[v][:-1]) / self.dy
        new[3] -= G * (xa[0][:, 1:] + xb[0][:, :-1]) * 0.5 * (xa[3][:, 1:] - xb[3][:, :-1]) / self.dx
        new[6] -= G * (ya[0][1:] + yb[0][:-1]) * 0.5 * (ya[3][1:] - yb[3][:-1]) / self.dy
        new[0] += self.sources(t)
        return new

    def fv_step(self, u, t, dt):
        def still(a):
            a = a.clone()
            a[3], a[6] = torch.where(a[0] > TOL, a[3], 0.0 * a[3]), torch.where(a[0] > TOL, a[6], 0.0 * a[6])
            return a

        u = self.friction(u, dt)
        v = still(u + dt * self.fv_operator(u, t))
        if self.scheme == "fv1":
            return v
        return still(0.5 * (u + v + dt * self.fv_operator(v, t + dt)))

    def step(self, u, t, dt):
        return self.dg2_step(u, t, dt) if self.scheme == "dg2" else self.fv_step(u, t, dt)

    def courant(self, u):
        wet = u[0] > TOL
        a, b = speeds(u[0], u[3], u[6])
        c = root(G * u[0])
        rate = torch.maximum((a.abs() + c) / self.dx, (b.abs() + c) / self.dy)
        r = float(torch.where(wet, rate, torch.zeros_like(rate)).max())
        return min(self.cfl / r, self.site.dt_max) if r > 0.0 else self.site.dt_max

    def depths(self, u):
        got = []
        for x, y in self.site.gauges:
            i, j = min(max(int(x / self.dx), 0), self.nx - 1), min(max(int(y / self.dy), 0), self.ny - 1)
            a, b = (x - (i + 0.5) * self.dx) / (0.5 * self.dx), (y - (j + 0.5) * self.dy) / (0.5 * self.dy)
            got.append(pos(u[0, j, i] + a * u[1, j, i] + b * u[2, j, i]))
        return torch.stack(got)

    def run_to(self, u, t, t_end):
        every, rows = self.site.sample_every, []
        nxt = (math.floor(t / every + 1e-9) + 1.0) * every
        while t < t_end:
            dt, target = self.courant(u), min(nxt, t_end)
            land = t + dt >= target
            dt = target - t if land else dt
            u = self.step(u, t, dt)
            t = target if land else t + dt
            if land and target == nxt:
                rows.append(self.depths(u).cpu().numpy())
                nxt += every
        return u, np.array(rows).reshape(-1, len(self.site.gauges))


def exact_run(case, site, t0, seed):
    p = Plain(site, case["scheme"], case["limiter"])
    u = p.put(water(site, seed, case["scheme"] != "dg2"))
    if case["kind"] == "steps":
        dt, t = 0.02 + 0.01 * random.Random(seed).random(), t0
        for _ in range(case["steps"]):
            u, t = p.step(u, t, dt), t + dt
        rows = np.zeros((0, len(site.gauges)))
    else:
        u, rows = p.run_to(u, t0, t0 + case["seconds"])
    got = {"state": u.cpu().numpy(), "gauges": rows}
    if not case["fp32"]:
        # the ledger closes on the mass
        m = float(u[0].sum()) * site.dx * site.dy
        got["mass"] = np.array([m, m])
    return got


def exact_gradient(case, seed):
    site, dts, samples, obs, man, q = calibration(case, seed)
    p = Plain(site)
    n, qk = p.put(man).requires_grad_(), p.put(q).requires_grad_()
    face, width, tk, _ = p.inflow
    h = modes(site.eta_corner - site.z_corner)
    start = np.zeros((9, site.ny, site.nx))
    start[:3] = np.where(h[0] > 0.0, np.stack(h), 0.0)
    seen = {k: p.put(o) for k, o in zip(samples, obs)}

    def advance(u, n_, q_, t, dt):
        p.n, p.inflow = n_, (face, width, tk, q_)
        return p.step(u, t, dt)

    us, t = [p.put(start)], 0.0
    times = []
    loss = 0.0
    with torch.no_grad():
        for k, dt in enumerate(dts):
            times.append(t)
            us.append(advance(us[-1], n, qk, t, float(dt)))
            t += float(dt)
            if k + 1 in seen:
                loss += float(((p.depths(us[-1]) - seen[k + 1]) ** 2).sum())
    back, gn, gq = torch.zeros_like(us[0]), torch.zeros_like(n), torch.zeros_like(qk)
    for k in range(len(dts) - 1, -1, -1):
        u = us[k].clone().requires_grad_()
        with torch.enable_grad():
            v = advance(u, n, qk, times[k], float(dts[k]))
            out = (v * back).sum()
            if k + 1 in seen:
                out = out + ((p.depths(v) - seen[k + 1]) ** 2).sum()
            a, b, c = torch.autograd.grad(out, (u, n, qk), allow_unused=True)
        back, gn, gq = a, gn + b, gq + (0.0 if c is None else c)
    return {"loss": np.array([loss]), "by_manning": gn.cpu().numpy(), "by_knot": gq.cpu().numpy()}


def exact(case, seed):
    if case["kind"] == "adjoint":
        return exact_gradient(case, seed)
    with torch.no_grad():
        if case["kind"] == "ensemble":
            return [exact_run(case, c, 600.0, seed + s) for s, c in enumerate(members_of(case, seed))]
        site, t0 = site_of(case, seed)
        return exact_run(case, site, t0, seed)
