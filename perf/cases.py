"""The work that users of this framework have it do, as cases that can be timed.

Each case is one piece of a simulation run through the public entry points:
a stretch of coupled time steps and the read-out that goes with it.  Sizes,
boundaries and parameters are those of configs/*.json, of the protocols and
of the tests; `draw` spreads them over the ranges they stand for.

`exact` holds a plain torch FP64 statement of the same steps (whole-field
operations, transformation matrices written out), which shares no code with
the library.
"""
import math

import numpy as np
import torch

import paper_2205_00686_gb300 as lbm
from paper_2205_00686_gb300 import workloads as W

TC = W.TC


# ---- cases -------------------------------------------------------------------

def listed():
    return [
        # the 64 x 64 parity configuration in FP64: the smallest domain anyone
        # runs; a step is all latency
        dict(name="static_64_fp64", kind="static", nx=64, ny=64, prec="fp64", steps=100),
        # the evaporation configuration: 20 000 steps on 256 x 256, advanced
        # in stretches with the fields read after each
        dict(name="open_256_fp32", kind="open", nx=256, ny=256, R=40.0, T_edge=0.95,
             prec="fp32", steps=200),
        # the D^2 law of Section 4.1 in FP64: periodic flow, temperature held
        # at the edges, the droplet's diagnostics sampled after each stretch
        dict(name="d2_200_fp64", kind="d2", nx=200, ny=200, R=30.0, T_edge=1.0, prec="fp64",
             steps=100, read="diagnostics"),
        # the heated-surface configuration with FP16-stored thermal
        # populations: a short run from its initial fields to its final
        # fields, with the contact angle
        dict(name="heated_400x200_g16", kind="heated", nx=400, ny=200, R=50.0, prec="fp32_g16",
             steps=200, fresh=True, read="angle"),
        # nucleate boiling with buoyancy and a heater: the start of a run and
        # the vapour regions that a departure watch looks at every 200 steps
        dict(name="boiling_300x600_fp32", kind="boiling", nx=300, ny=600, gravity=2e-5,
             prec="fp32", steps=200, fresh=True, read="regions"),
        # the throughput workload
        dict(name="open_4096_fp32", kind="open", nx=4096, ny=4096, R=640.0, T_edge=0.95,
             prec="fp32", steps=50),
        # a large FP64 run of ragged size (the reference runs that FP32 is
        # judged against)
        dict(name="open_1999x1501_fp64", kind="open", nx=1999, ny=1501, R=400.0, T_edge=0.95,
             prec="fp64", steps=10),
        # many independent droplets of uneven size in one batch (the batched
        # and served population), advanced together and read back
        dict(name="batch_64_fp32", kind="batch", count=64, side_lo=64, side_hi=512, prec="fp32",
             steps=150),
        # the interface analyses on a large field: diagnostics and the vapour
        # regions of a pool full of bubbles
        dict(name="bubbles_2048_fp32", kind="bubbles", nx=2048, ny=2048, prec="fp32", steps=0,
             read="analysis"),
        # the three-dimensional throughput workload and its fields
        dict(name="cloud_256_fp32", kind="cloud3", nx=256, ny=256, nz=256, cells=4, prec="fp32",
             steps=100),
        # a droplet between heated walls in three dimensions with buoyancy, a
        # small ragged box, from its initial fields to its final ones
        dict(name="walls_72x50x61_fp32", kind="walls3", nx=72, ny=50, nz=61, R=12.0,
             gravity=1e-5, prec="fp32", steps=100, fresh=True),
        # the three-dimensional form in FP64
        dict(name="cloud_96_fp64", kind="cloud3", nx=96, ny=96, nz=96, cells=3, prec="fp64",
             steps=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps(nodes, budget, most):
    return int(max(8, min(most, budget // nodes)))


def draw(rng):
    kind = rng.choice(["open", "open", "open", "static", "d2", "heated", "boiling", "batch",
                       "bubbles", "cloud3", "walls3"])
    if kind in ("open", "static", "d2"):
        prec = rng.choice(["fp32", "fp32", "fp64", "fp32_g16"])
        nx = _log(rng, 56, 1400 if prec == "fp64" else 3600)
        ny = max(56, int(nx * rng.uniform(0.6, 1.2)))
        c = dict(kind=kind, nx=nx, ny=ny, R=round(rng.uniform(0.2, 0.3) * min(nx, ny), 2),
                 prec=prec, steps=_steps(nx * ny, 2e7 if prec == "fp64" else 4e8, 200), fresh=True)
        if kind == "d2":
            c.update(T_edge=1.0)
            if prec != "fp32_g16" and rng.random() < 0.5:
                c.update(read="diagnostics")
        elif kind == "open":
            c.update(T_edge=round(rng.uniform(0.90, 0.98), 4))
        return c
    if kind == "heated":
        nx = _log(rng, 120, 1600)
        return dict(kind=kind, nx=nx, ny=int(nx * rng.uniform(0.4, 0.7)), R=round(nx / 8.0, 2),
                    prec=rng.choice(["fp32", "fp32_g16"]), steps=rng.randrange(100, 201),
                    fresh=True, read="angle")
    if kind == "boiling":
        nx = _log(rng, 120, 900)
        return dict(kind=kind, nx=nx, ny=int(nx * rng.uniform(1.2, 2.2)),
                    gravity=rng.choice([1e-5, 2e-5, 4e-5, 8e-5]), prec="fp32", steps=200,
                    fresh=True, read="regions")
    if kind == "batch":
        return dict(kind=kind, count=_log(rng, 6, 72), side_lo=64, side_hi=rng.randrange(160, 513),
                    prec=rng.choice(["fp32", "fp32", "fp32_g16"]), steps=rng.randrange(64, 151))
    if kind == "bubbles":
        nx = _log(rng, 300, 2600)
        return dict(kind=kind, nx=nx, ny=int(nx * rng.uniform(0.5, 1.5)), prec="fp32", steps=0,
                    read="analysis")
    prec = rng.choice(["fp32", "fp32", "fp64"])
    if kind == "cloud3":
        cells = rng.choice([1, 2, 3, 4])
        n = cells * rng.randrange(28, 57 if prec == "fp32" else 33)
        return dict(kind=kind, nx=n, ny=n, nz=n, cells=cells, prec=prec,
                    steps=_steps(n ** 3, 4e8 if prec == "fp32" else 2e7, 100))
    nx, ny, nz = (rng.randrange(36, 110 if prec == "fp32" else 64) for _ in range(3))
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, R=round(0.25 * min(nx, ny, nz, 64), 2),
                gravity=rng.choice([0.0, 1e-5]), prec=prec,
                steps=_steps(nx * ny * nz, 2e8 if prec == "fp32" else 2e7, 100), fresh=True)


def _members(case):
    """Sides, relative radii and edge temperatures of a batch's domains: fixed
    by the case, so that every seed has the same work."""
    u = np.random.RandomState(1000 * case["count"] + case["side_hi"]).rand(case["count"], 3)
    lo, hi = case["side_lo"], case["side_hi"]
    return [dict(kind="open", nx=lo + int(a * (hi - lo + 1)), ny=lo + int(a * (hi - lo + 1)),
                 R=(0.2 + 0.1 * b) * (lo + int(a * (hi - lo + 1))), T_edge=0.90 + 0.08 * t,
                 prec=case["prec"]) for a, b, t in u]


# ---- inputs -----------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _noise(shape, amp, gen):
    return amp * (2.0 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64) - 1.0)


def _axis(n):
    return torch.arange(n, device="cuda", dtype=torch.float64)


def _tanh(d, R, w, inside, outside):
    return 0.5 * (inside + outside) - 0.5 * (inside - outside) * torch.tanh((d - R) / (0.5 * w))


def _inputs(case, seed):
    """Parameters, boundaries, rho and T (FP64, on the GPU) of one domain; the
    velocity is zero.  The seed moves the droplet by up to a node and draws
    the noise."""
    gen = _gen(seed)
    kind = case["kind"]
    rg, rl = W.COEXISTENCE[0.86]
    Ts = 0.86 * TC
    off = [float(v) for v in _noise(3, 1.0, gen).cpu()]
    nx, ny = case["nx"], case["ny"]
    if kind in ("cloud3", "walls3"):
        nz = case["nz"]
        z, y, x = _axis(nz)[:, None, None], _axis(ny)[None, :, None], _axis(nx)[None, None, :]
        p = W.params(gravity=case.get("gravity", 0.0))
        if kind == "cloud3":
            s = nx // case["cells"]
            c = 0.5 * (s - 1)
            d = torch.sqrt((x % s - c) ** 2 + (y % s - c) ** 2 + (z % s - c) ** 2)
            rho = _tanh(d, 0.25 * s, 4.0, rl, rg)
            T = torch.full_like(rho, Ts)
            bc = W.periodic_bc3()
        else:
            d = torch.sqrt((x - 0.5 * (nx - 1) - off[0]) ** 2 + (y - 0.5 * (ny - 1) - off[1]) ** 2
                           + (z - 0.5 * (nz - 1) - off[2]) ** 2)
            rho = _tanh(d, case["R"], 4.0, rl, rg)
            T = _tanh(d, case["R"], 4.0, Ts, 0.95 * TC)
            bc = W.wall_bc3(0.95 * TC, 0.95 * TC)
        return dict(p=p, bc=bc, rho=rho + _noise(rho.shape, 1e-4, gen), T=T)
    y, x = _axis(ny)[:, None], _axis(nx)[None, :]
    p = W.params()
    if kind in ("static", "open", "d2"):
        R = case.get("R", 0.25 * nx)
        d = torch.sqrt((x - 0.5 * (nx - 1) - off[0]) ** 2 + (y - 0.5 * (ny - 1) - off[1]) ** 2)
        rho = _tanh(d, R, 4.0, rl, rg)
        if kind == "static":
            T = torch.full_like(rho, Ts)
            bc = W.periodic_bc()
        else:
            Te = case["T_edge"] * TC
            T = _tanh(d, R, 4.0, Ts, Te)
            bc = W.bc_spec([W.OPEN if kind == "open" else W.PERIODIC] * 4, [W.T_DIRICHLET] * 4,
                           T_edge=[Te] * 4)
        return dict(p=p, bc=bc, rho=rho + _noise(rho.shape, 1e-4, gen), T=T)
    flow = [W.PERIODIC, W.PERIODIC, W.WALL, W.OPEN]
    therm = [W.T_PERIODIC, W.T_PERIODIC, W.T_DIRICHLET, W.T_DIRICHLET]
    if kind == "heated":
        p = W.params(lambda_=0.08)
        d = torch.sqrt((x - 0.5 * nx - off[0]) ** 2 + y ** 2)
        rho = _tanh(d, case["R"], 5.0, rl, rg) + _noise((ny, nx), 1e-4, gen)
        bc = W.bc_spec(flow, therm, T_edge=[0.0, 0.0, 0.95 * TC, Ts], theta_deg=90.0)
    elif kind == "boiling":
        p = W.params(lambda_=2.0 / 3.0, gravity=case["gravity"])
        rho = rl + _noise((ny, nx), 1e-3, gen)
        x0 = nx // 2 - 10
        bc = W.bc_spec(flow, therm, T_edge=[0.0, 0.0, Ts, Ts], theta_deg=75.0,
                       heater=(x0, x0 + 20), T_heater=1.1 * TC)
    else:   # bubbles: one in each cell of a jittered grid, away from its edges
        p = W.params(lambda_=2.0 / 3.0, gravity=2e-5)
        s = _CELL
        my, mx = -(-ny // s), -(-nx // s)
        r = torch.rand((3, my, mx), generator=gen, device="cuda", dtype=torch.float64)
        R = 10.0 + 20.0 * r[0]
        cy = 0.5 * s + (2.0 * r[1] - 1.0) * (0.5 * s - 8.0 - R)
        cx = 0.5 * s + (2.0 * r[2] - 1.0) * (0.5 * s - 8.0 - R)
        iy, ix = (y // s).long(), (x // s).long()
        d = torch.sqrt((x % s - cx[iy, ix]) ** 2 + (y % s - cy[iy, ix]) ** 2)
        rho = _tanh(d - R[iy, ix], 0.0, 4.0, rg, rl) + _noise((ny, nx), 1e-3, gen)
        bc = W.bc_spec(flow, therm, T_edge=[0.0, 0.0, Ts, Ts], theta_deg=75.0)
    return dict(p=p, bc=bc, rho=rho, T=torch.full_like(rho, Ts))


def _domain(case, inp):
    """The context and the host fields it starts from."""
    rho, T = inp["rho"].cpu().numpy(), inp["T"].cpu().numpy()
    zero = np.zeros_like(rho)
    if rho.ndim == 3:
        d = lbm.Domain3(case["nx"], case["ny"], case["nz"], inp["p"], inp["bc"], prec=case["prec"])
        host = (rho, zero, zero, zero, T)
    else:
        d = lbm.Domain(case["nx"], case["ny"], inp["p"], inp["bc"], prec=case["prec"])
        host = (rho, zero, zero, T)
    d.init_fields(*host)
    return d, host


def prepare(case, seed):
    if case["kind"] == "batch":
        st = dict(case=case, batch=lbm.Batch(), doms=[], outs=[])
        ms = _members(case)
        st["buf"] = torch.empty(sum(4 * m["nx"] * m["ny"] for m in ms), dtype=torch.float64,
                                pin_memory=True)
        at = 0
        for k, m in enumerate(ms):
            d, _ = _domain(m, _inputs(m, 1009 * seed + k))
            st["doms"].append(d)
            st["batch"].attach(d)
            n = m["nx"] * m["ny"]
            st["outs"].append(tuple(st["buf"][at + q * n: at + (q + 1) * n].view(m["ny"], m["nx"])
                                    for q in range(4)))
            at += 4 * n
        return st
    d, host = _domain(case, _inputs(case, seed))
    st = dict(case=case, d=d, host=host if case.get("fresh") else None)
    if _fields_out(case):
        st["buf"] = torch.empty((len(host),) + host[0].shape, dtype=torch.float64, pin_memory=True)
    elif case.get("read") != "analysis":
        dt = torch.float64 if case["prec"] == "fp64" else torch.float32
        st["buf"] = torch.empty(d.rows_bytes(case["ny"]) // dt.itemsize, dtype=dt, device="cuda")
    return st


def _fields_out(case):
    """FP16-stored populations, batches, three dimensions and FP32 domains of
    the sizes one looks at give their fields (in the precision they were
    computed in); FP64 and the large FP32 domains hand on their packed state."""
    if case["prec"] == "fp32_g16" or case["kind"] in ("batch", "cloud3", "walls3"):
        return True
    return case["prec"] == "fp32" and case["nx"] * case["ny"] <= 1 << 20


# ---- one pass -----------------------------------------------------------------

_DIAG = ("mass", "energy", "liquid_mass", "liquid_area", "liquid_area_smooth", "diameter",
         "diameter_smooth", "max_u")
_ANGLE = ("theta_deg", "xc", "yc", "radius", "base_width", "height")
_REGION = ("label", "area", "sum_y", "y_min", "y_max", "touches_w", "touches_e", "touches_s",
           "touches_n")


_CELL = 96   # side of the cells of the bubble field, one bubble in each


def _most_regions(case):
    return (case["nx"] // _CELL + 1) * (case["ny"] // _CELL + 1)


def _levels():
    rg, rl = W.COEXISTENCE[0.86]
    return rl, rg


def run(state):
    case = state["case"]
    rl, rg = _levels()
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        for d, o in zip(state["doms"], state["outs"]):
            d.get_rho_u_T(o)
        return dict(fields=state["buf"].float())
    d = state["d"]
    if state["host"] is not None:
        d.init_fields(*state["host"])
    d.step(case["steps"])
    out = {}
    read = case.get("read")
    real = np.float64 if case["prec"] == "fp64" else np.float32
    if read in ("diagnostics", "analysis"):
        v = d.diagnostics(rl, rg)
        out["diagnostics"] = np.array([v[k] for k in _DIAG], real)
    if read in ("regions", "analysis"):
        v = d.regions(0.5 * (rl + rg), below=True)
        # one row for each region found, in a table long enough for any seed
        table = np.full((_most_regions(case), len(_REGION)), -1, np.int64)
        for row, r in zip(table, v):
            row[:] = [r[k] for k in _REGION]
        out["regions"] = table
    if read == "angle":
        v = d.contact_angle(rl, rg)
        out["angle"] = np.array([v[k] for k in _ANGLE], real)
    if read == "analysis":
        return out
    if _fields_out(case):
        if case["kind"] in ("cloud3", "walls3"):
            d.get_fields(tuple(state["buf"]))
        else:
            d.get_rho_u_T(tuple(state["buf"]))
        out["fields"] = state["buf"].clone() if case["prec"] == "fp64" else state["buf"].float()
    else:
        d.pack_rows(0, case["ny"], state["buf"].data_ptr())
        out["state"] = state["buf"]
    return out


# ---- what a pass cannot do without ----------------------------------------------

def _nodes(case):
    if case["kind"] == "batch":
        return sum(m["nx"] * m["ny"] for m in _members(case))
    return case["nx"] * case["ny"] * case.get("nz", 1)


def work(case):
    """Each step reads the state (f, g and the P history) once and writes it
    once; the read-out reads the state once and writes what it returns."""
    n, prec = _nodes(case), case["prec"]
    three = case["kind"] in ("cloud3", "walls3")
    ef, eg = (8, 8) if prec == "fp64" else (4, 2 if prec == "fp32_g16" else 4)
    node = 27 * ef if three else 10 * ef + 5 * eg
    read = (5 if three else 4) * 8 if _fields_out(case) else node
    if case.get("read") == "analysis":
        read = 0
    # operations a node update cannot do without (moments, EOS, force stencil,
    # two collisions, blend), from the counted FP64 step in two dimensions
    flops = 700 if three else 300
    return dict(bytes=n * (2 * node * case["steps"] + node + read),
                flops=n * (flops * case["steps"] + 40))


# ---- the same pass in plain FP64 --------------------------------------------------

def _eos(p, rho, T):
    """psi^2 and T (dp/dT)_rho of the Peng-Robinson EOS."""
    a, b, R, om = p["a"], p["b"], p["R"], p["omega"]
    k = 0.37464 + 1.54226 * om - 0.26992 * om * om
    Tc = 0.0778 * a / (0.45724 * b * R)
    s = torch.sqrt(T / Tc)
    h = 1.0 + k * (1.0 - s)
    den = 1.0 + 2.0 * b * rho - (b * rho) ** 2
    pr = rho * R * T / (1.0 - b * rho) - a * h * h * rho * rho / den
    dp = rho * R / (1.0 - b * rho) + a * k * h * rho * rho / (s * Tc * den)
    return 2.0 * (pr - rho / 3.0) / p["G"], T * dp


def _cuda(rows):
    return torch.tensor(rows, device="cuda", dtype=torch.float64)


class _Exact:
    """One domain in FP64; D2Q9 + D2Q5 or D3Q19 + D3Q7 by the number of axes.
    Axes are ordered as the fields are (y, x or z, y, x); velocities x first."""

    def __init__(self, inp):
        self.p, self.bc = inp["p"], inp["bc"]
        rho, T = inp["rho"], inp["T"]
        self.D = rho.dim()
        p, wd = self.p, self.p["w_dot"]
        e = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
        if self.D == 2:
            self.c = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
            self.h = self.c[:5]
            self.w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
            self.varpi = [0.0] + [1 / 3] * 4 + [1 / 12] * 4
            self.M = _cuda([[1] * 9, [-4] + [-1] * 4 + [2] * 4, [4] + [-2] * 4 + [1] * 4,
                            [v[0] for v in self.c], [0, -2, 0, 2, 0, 1, -1, -1, 1],
                            [v[1] for v in self.c], [0, 0, -2, 0, 2, 1, 1, -1, -1],
                            [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]])
            sp = 1.0 / (3.0 * p["nu"] + 0.5)
            self.S = [p["s0"], p["s_e"], p["s_eps"], p["s_j"], p["s_q"], p["s_j"], p["s_q"], sp, sp]
            self.Mh = _cuda([[1] * 5, [0, 1, 0, -1, 0], [0, 0, 1, 0, -1], [0, 1, 1, 1, 1],
                             [0, 1, -1, 1, -1]])
            self.cs2 = wd / 2.0
            flow, therm = self.bc["flow"], self.bc["therm"]
            self.flow = [(flow[2], flow[3]), (flow[0], flow[1])]     # y, x
            self.therm = [(therm[2], therm[3]), (therm[0], therm[1])]
            Te = self.bc["T_edge"]
            south = torch.full((rho.shape[1],), Te[2], device="cuda", dtype=torch.float64)
            south[self.bc["heater_x0"]:self.bc["heater_x1"]] = self.bc["T_heater"]
            self.Te = [(south, Te[3]), (Te[0], Te[1])]
        else:
            self.c = [(0, 0, 0)]
            for a in range(3):
                self.c += [e[a], tuple(-v for v in e[a])]
            for a, b in ((0, 1), (0, 2), (1, 2)):
                for s in (1, -1):
                    v = [0, 0, 0]
                    v[a], v[b] = 1, s
                    self.c += [tuple(v), tuple(-q for q in v)]
            self.h = self.c[:7]
            self.w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
            self.varpi = [0.0] + [1 / 6] * 6 + [1 / 12] * 12
            rows = []
            for x, y, z in self.c:
                q = x * x + y * y + z * z
                rows.append([1, 19 * q - 30, (21 * q * q - 53 * q + 24) / 2, x, (5 * q - 9) * x, y,
                             (5 * q - 9) * y, z, (5 * q - 9) * z, 3 * x * x - q,
                             (3 * q - 5) * (3 * x * x - q), y * y - z * z,
                             (3 * q - 5) * (y * y - z * z), x * y, y * z, x * z,
                             (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z])
            self.M = _cuda(rows).t().contiguous()
            sp, sq = 1.0 / (3.0 * p["nu"] + 0.5), p["s_q"]
            self.S = [p["s0"], p["s_e"], p["s_eps"], p["s_j"], sq, p["s_j"], sq, p["s_j"], sq, sp, sq,
                      sp, sq, sp, sp, sp, sq, sq, sq]
            self.Mh = _cuda([[1, x, y, z, x * x + y * y + z * z, x * x - y * y, y * y - z * z]
                             for x, y, z in self.h]).t().contiguous()
            self.cs2 = wd / 3.0
            fz = self.bc["flow_z"]
            self.flow = [(fz, fz), (W.PERIODIC,) * 2, (W.PERIODIC,) * 2]
            self.therm = [tuple(self.bc["therm"]), (W.T_PERIODIC,) * 2, (W.T_PERIODIC,) * 2]
            self.Te = [tuple(self.bc["T_edge"]), (0.0, 0.0), (0.0, 0.0)]
        n = len(self.h) - 1
        self.wh = [1.0 - wd] + [wd / n] * n
        self.opp = [self.c.index(tuple(-v for v in c)) for c in self.c]
        self.S = _cuda(self.S)
        vs1 = 1.0 / (p["lambda_"] / self.cs2 + 0.5)
        self.vs1 = vs1
        self.Lam = _cuda([p["vs0"]] + [vs1] * self.D + [p["vs3"]] + [p["vs4"]] * (self.D - 1))
        self.Minv, self.Mhinv = torch.linalg.inv(self.M), torch.linalg.inv(self.Mh)
        # u = 0 at the start: f^eq = w rho, g = w^ T
        self.f = torch.stack([w * rho for w in self.w])
        self.g = torch.stack([w * T for w in self.wh])
        self.P = torch.zeros_like(rho)
        self.n = 0
        self.rho_ref, self.T_ref = rho.mean(), T.mean()
        self.rho_ave = self.rho_ref

    def take(self, a, c, kinds, ghost=None):
        """a(x + c): periodic axes wrap, open ones repeat the edge, and beyond
        a wall of the first axis the ghost rows stand (0 without)."""
        for ax in range(self.D):
            s = c[self.D - 1 - ax]
            if s == 0:
                continue
            n = a.shape[ax]
            at = torch.arange(n, device="cuda") + s
            kind = kinds[ax][0 if s < 0 else 1]
            at = at % n if kind == W.PERIODIC else at.clamp(0, n - 1)
            a = a.index_select(ax, at)
        s = c[-1]
        if s and kinds[0][0 if s < 0 else 1] == W.WALL:
            # the row beyond the wall, with the shift along the other axes
            row = 0 if s < 0 else a.shape[0] - 1
            if ghost is None:
                a[row] = 0.0
            else:
                gr = ghost[0 if s < 0 else 1]
                for ax in range(1, self.D):
                    t = c[self.D - 1 - ax]
                    if t:
                        at = torch.arange(gr.shape[ax - 1], device="cuda") + t
                        n = gr.shape[ax - 1]
                        at = at % n if kinds[ax][0] == W.PERIODIC else at.clamp(0, n - 1)
                        gr = gr.index_select(ax - 1, at)
                a[row] = gr
        return a

    def macro(self):
        p, D, c = self.p, self.D, self.c
        f, g = self.f, self.g
        self.rho, self.T = f.sum(0), g.sum(0)
        q, self.tdp = _eos(p, self.rho, self.T)
        psi = torch.sqrt(q)
        ghost = [None, None]
        for e in range(2):
            if self.flow[0][e] != W.WALL:
                continue
            r1, r2 = (self.rho[0], self.rho[1]) if e == 0 else (self.rho[-1], self.rho[-2])
            d2 = 0.0
            for ax in range(D - 1):
                n = r1.shape[ax]
                i = torch.arange(n, device="cuda")
                per = self.flow[ax + 1][0] == W.PERIODIC
                hi = (i + 1) % n if per else (i + 1).clamp(0, n - 1)
                lo = (i - 1) % n if per else (i - 1).clamp(0, n - 1)
                d2 = d2 + (r1.index_select(ax, hi) - r1.index_select(ax, lo)) ** 2
            th = math.tan(math.pi / 2.0 - math.radians(self.bc["theta_deg"]))
            ghost[e] = torch.sqrt(_eos(p, r2 + th * torch.sqrt(d2), self.T[0 if e == 0 else -1])[0])
        s = [torch.zeros_like(psi) for _ in range(D)]
        for i in range(1, len(c)):
            pn = self.take(psi, c[i], self.flow, ghost)
            for a in range(D):
                if c[i][a]:
                    s[a] += (self.varpi[i] * c[i][a]) * pn
        self.F = [-p["G"] * psi * v for v in s]
        self.Fm2 = p["G"] ** 2 * sum(v * v for v in s)     # |F_m|^2 / psi^2
        self.F[D - 1] = self.F[D - 1] - p["gravity"] * (self.rho - self.rho_ave)
        self.u = []
        for a in range(D):
            j = sum(c[i][a] * f[i] for i in range(len(c)) if c[i][a])
            self.u.append((j + 0.5 * self.F[a]) / self.rho)

    def step(self):
        p, D, c, w = self.p, self.D, self.c, self.w
        self.macro()
        rho, u, F = self.rho, self.u, self.F
        div = torch.zeros_like(rho)
        for i in range(1, len(c)):
            for a in range(D):
                if c[i][a]:
                    div += (3.0 * w[i] * c[i][a]) * self.take(u[a], c[i], self.flow)
        shape = rho.shape
        mh = (self.Mh @ self.g.reshape(len(self.h), -1)).reshape((-1,) + shape)
        C = rho * p["cv"]
        Q = -(C * sum(u[a] * (-self.vs1 / self.cs2) * mh[1 + a] for a in range(D)) + self.tdp * div)
        Pn = Q / C
        Qs = Q if self.n == 0 else Q + 0.5 * C * (Pn - self.P)
        # D2Q9 / D3Q19: equilibrium and discrete force in velocity space, then
        # relaxation in moment space, with the sigma terms of Eq. 8
        uu, uF = sum(v * v for v in u), sum(u[a] * F[a] for a in range(D))
        feq, fF = torch.empty_like(self.f), torch.empty_like(self.f)
        for i in range(len(c)):
            cu = sum(c[i][a] * u[a] for a in range(D)) if any(c[i]) else torch.zeros_like(rho)
            cF = sum(c[i][a] * F[a] for a in range(D)) if any(c[i]) else torch.zeros_like(rho)
            feq[i] = w[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu)
            fF[i] = w[i] * (3.0 * cF - 3.0 * uF + 9.0 * cu * cF)
        nq = len(c)
        meq = self.M @ feq.reshape(nq, -1)
        mF = self.M @ fF.reshape(nq, -1)
        if D == 2:   # m^eq of Eq. 7 and the force moments of Eq. 8, as printed
            meq[2] = (rho - 3.0 * rho * uu).reshape(-1)
            mF[2] = -(6.0 * uF).reshape(-1)
            sig = p["sigma"] * self.Fm2.reshape(-1)
            mF[1] += sig / (1.0 / p["s_e"] - 0.5)
            mF[2] -= sig / (1.0 / p["s_eps"] - 0.5)
        else:
            mF[1] += 9.5 * p["sigma"] * self.Fm2.reshape(-1) / (1.0 / p["s_e"] - 0.5)
        m = self.M @ self.f.reshape(nq, -1)
        S = self.S[:, None]
        fs = (self.Minv @ (m - S * (m - meq) + (1.0 - 0.5 * S) * mF)).reshape(self.f.shape)
        del m, meq, mF, feq, fF
        fn = torch.empty_like(fs)
        for i in range(nq):
            back = tuple(-v for v in c[i])
            fn[i] = self.take(fs[i], back, self.flow)
            for e, row in ((0, 0), (1, -1)):
                if self.flow[0][e] == W.WALL and c[i][-1] == (1 if e == 0 else -1):
                    fn[i][row] = fs[self.opp[i]][row]
        # D2Q5 / D3Q7
        nh = len(self.h)
        mh = mh.reshape(nh, -1)
        one = torch.zeros(nh, 1, device="cuda", dtype=torch.float64)
        one[0], one[D + 1] = 1.0, p["w_dot"]
        mheq = one * self.T.reshape(1, -1)
        gs = (self.Mhinv @ (mh - self.Lam[:, None] * (mh - mheq) + one * Qs.reshape(1, -1)))
        gs = gs.reshape(self.g.shape)
        per = [(W.PERIODIC, W.PERIODIC)] * D
        gn = torch.empty_like(gs)
        for i in range(nh):
            back = tuple(-v for v in c[i])
            A = self.take(gs[i], back, per)
            for ax in range(D):
                s = back[D - 1 - ax]
                if s == 0:
                    continue
                e = 0 if s < 0 else 1
                kind = self.therm[ax][e]
                if kind == W.T_PERIODIC:
                    continue
                own = gs[self.opp[i]].select(ax, 0 if e == 0 else -1)
                if kind == W.T_DIRICHLET:
                    own = 2.0 * self.wh[i] * self.Te[ax][e] - own
                A.select(ax, 0 if e == 0 else A.shape[ax] - 1).copy_(own)
            gn[i] = self.g[i] + (A - self.g[i]) / C
        self.f, self.g, self.P = fn, gn, Pn
        self.rho_ave = rho.mean()
        self.n += 1

    def packed(self):
        w, wh = _cuda(self.w), _cuda(self.wh)
        ones = (1,) * self.D
        return torch.cat([(self.f - w.view(-1, *ones) * self.rho_ref).reshape(-1),
                          (self.g - wh.view(-1, *ones) * self.T_ref).reshape(-1),
                          self.P.reshape(-1)])

    def fields(self):
        self.macro()
        return torch.stack([self.rho] + self.u + [self.T])

    def diagnostics(self, rl, rg):
        r, u, T = (lambda v: (v[0], v[1:-1], v[-1]))(self.fields())
        liq = r > 0.5 * (rl + rg)
        area = float(liq.sum())
        smooth = float(((r - rg) / (rl - rg)).clamp(0.0, 1.0).sum())
        return np.array([float(r.sum()), float((r * self.p["cv"] * T).sum()), float(r[liq].sum()),
                         area, smooth, math.sqrt(4.0 / math.pi * area),
                         math.sqrt(4.0 / math.pi * smooth), float((u * u).sum(0).max().sqrt())])


def exact(case, seed):
    if case["kind"] == "batch":
        parts = []
        for k, m in enumerate(_members(case)):
            e = _Exact(_inputs(m, 1009 * seed + k))
            for _ in range(case["steps"]):
                e.step()
            parts.append(e.fields().reshape(-1))
        return dict(fields=torch.cat(parts))
    e = _Exact(_inputs(case, seed))
    for _ in range(case["steps"]):
        e.step()
    rl, rg = _levels()
    read = case.get("read")
    out = {}
    if read in ("diagnostics", "analysis"):
        out["diagnostics"] = e.diagnostics(rl, rg)
    if read in ("regions", "analysis"):
        out["regions"] = None
    if read == "angle":
        out["angle"] = None
    if read != "analysis":
        if _fields_out(case):
            out["fields"] = e.fields()
        else:
            out["state"] = e.packed()
    return out
