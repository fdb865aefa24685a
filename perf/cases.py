"""What a user has this library do, as cases that can be timed: marching jets in each precision and mesh form, a
batch of jets, a monitored run, a host-coupled step, the device-side sums, and the far-field evaluation.

A case is a dict of plain values; `prepare` makes what a program has in hand before the call, `run` is one pass
through the public entry points (paper_2212_12365_gb300.les and the C ABI it binds), `work` counts what the pass
cannot do without, and `exact` gives the same outputs from a plain 64-bit torch statement of the method.
"""
import ctypes
import functools
import math

import numpy as np
import torch

from paper_2212_12365_gb300 import inputs as I
from paper_2212_12365_gb300 import les

DEV = "cuda"
PREC = {"fp64": les.LES_FP64, "fp32": les.LES_FP32, "fp32-sep": les.LES_FP32_SEPARABLE}
ALPHA = (1 / 4, 1 / 6, 3 / 8, 1 / 2, 1.0)


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------

def _march(name, mesh, n, prec, steps, **kw):
    c = {"do": "march", "mesh": mesh, "ni": n[0], "nj": n[1], "nk": n[2], "prec": prec, "steps": steps,
         "mach": 1.4, "TR": 1.0, "probe": 0, "monitor": 0, "exchange": 0}
    c.update(kw)
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest jet, FP64: 49k points, ten steps and the state back (launches and latency count)
        _march("fp64-jet-48x32x32", "jet", (48, 32, 32), "fp64", 10),
        # the paper-scale single jet (14.2 M points) in FP64, the form a production run marches in
        _march("fp64-jet-384x256x144", "jet", (384, 256, 144), "fp64", 4),
        # one of the paper's own mesh sizes on its polar topology with the centerline, FP64, ragged sizes
        _march("fp64-polar-200x75x40", "polar", (200, 75, 40), "fp64", 10),
        # the same paper-scale jet in FP32: forty steps between snapshots
        _march("fp32-jet-384x256x144", "jet", (384, 256, 144), "fp32", 40),
        # and with the separable-metric option, which a user of a product grid may ask for
        _march("fp32sep-jet-384x256x144", "jet", (384, 256, 144), "fp32-sep", 40),
        # the large jet (56.6 M points, TR 2) with the cylinder probe that feeds the far field, every 5 steps
        _march("fp32-jet-768x384x192-probe", "jet", (768, 384, 192), "fp32", 10, TR=2.0, probe=5),
        # the paper's polar mesh, FP32: the general curvilinear form with the centerline (3.6 M points)
        _march("fp32-polar-400x150x60", "polar", (400, 150, 60), "fp32", 40),
        # 64 independent jets of uneven sizes, Mach numbers and temperature ratios in one handle
        {"name": "fp32-batch-64", "do": "batch", "jets": 64, "draw": 4, "prec": "fp32", "steps": 10},
        # a small jet coupled to a host program: state in, one step, state out (latency)
        _march("fp32-jet-48x32x32-exchange", "jet", (48, 32, 32), "fp32", 1, exchange=1),
        # a mid-size run watched by the residual monitor every ten steps
        _march("fp32-jet-192x128x72-monitor", "jet", (192, 128, 72), "fp32", 50, monitor=10),
        # residual and conservation sums of a caller's own device buffers at the paper-scale size
        {"name": "sums-14155776", "do": "sums", "points": 384 * 256 * 144},
        # far field of the large jet's probe cylinder: 64 microphones x 512 times from 1024 frames
        {"name": "fwh-256x384-64x512", "do": "fwh", "n_theta": 256, "n_x": 384, "frames": 1024, "mics": 64,
         "times": 512, "dt_ratio": 1.0},
    ]


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same kinds; sizes over the logarithm of their range, odd ones among them."""
    kind = rng.choice(["jet", "jet", "jet", "polar", "batch", "sums", "fwh"])
    if kind == "sums":
        return {"do": "sums", "points": int(_logu(rng, 1e4, 1.4e7))}
    if kind == "batch":
        return {"do": "batch", "jets": rng.randint(2, 24), "draw": rng.randint(5, 10 ** 6),
                "prec": rng.choice(["fp32", "fp32-sep", "fp64"]), "steps": rng.randint(2, 6)}
    if kind == "fwh":
        return {"do": "fwh", "n_theta": rng.randint(48, 256), "n_x": rng.randint(40, 300),
                "frames": rng.randint(800, 1024), "mics": rng.randint(1, 64), "times": rng.randint(40, 512),
                "dt_ratio": rng.choice([0.5, 1.0, rng.uniform(0.3, 1.0)])}
    prec = rng.choice(["fp64", "fp32"] if kind == "polar" else ["fp64", "fp32", "fp32-sep"])
    pts = _logu(rng, 3e4, 2.5e6 if prec == "fp64" else 8e6)
    # aspect ratios of the configurations: axial longest, azimuthal / spanwise shortest
    a, b = rng.uniform(1.2, 3.0), rng.uniform(0.4, 1.0)
    nj = max(16, round((pts / (a * b)) ** (1 / 3)))
    ni, nk = max(24, round(a * nj)), max(12, round(b * nj))
    n = ni * nj * nk
    steps = max(2, min(40, round((3e6 if prec == "fp64" else 4e7) / n)))
    extra = rng.choice([{}, {}, {"monitor": max(1, steps // 2)}, {"exchange": 1}])
    if kind == "jet" and rng.random() < 0.3:
        extra = {"probe": rng.randint(1, 3)}
    return _march(None, kind, (ni, nj, nk), prec, steps, mach=rng.uniform(1.2, 2.0), TR=rng.uniform(1.0, 3.0),
                  **extra)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=12)
def _grid(mesh, ni, nj, nk):
    """The mesh of a case (the same for every seed)."""
    if mesh == "polar":
        return I.polar_jet_grid(ni, nj, nk, 30.0, 12.0)
    if mesh == "small":  # the smallest configuration: 8 points across the jet diameter
        return I.jet_grid(ni, nj, nk, 20.0, 10.0, 10.0, 1 / 8, 1 / 8)
    return I.jet_grid(ni, nj, nk, 30.0, 12.0, 12.0, 0.4 * 12.0 / (nj - 1), 0.4 * 12.0 / (nk - 1))


def _spec(c):
    small = c["mesh"] == "jet" and c["ni"] * c["nj"] * c["nk"] < 60000
    return _grid("small" if small else c["mesh"], c["ni"], c["nj"], c["nk"])


def _flow(c, seed):
    return I.FlowParams(mach_j=c["mach"], TR=c["TR"], Re=1.0e5, Cs=0.17, cfl=0.5, seed=seed + 1)


def _jet_state(spec, fp, seed):
    """A developed jet to start from, primitives [5][N] in FP64 on the GPU: the entrance profile carried downstream
    in a spreading shear layer, with smooth seeded disturbances of a few per cent in and around the layer.  The far
    faces hold the ambient at rest, as they do in a jet run: the far-field condition changes branch with the sign
    of the normal velocity, which there is zero up to weak waves."""
    rng = np.random.default_rng([seed, spec.N])
    ni, nj, nk = spec.dims
    x, y, z = (torch.as_tensor(v, device=DEV).view(nk, nj, ni) for v in (spec.x, spec.y, spec.z))
    r = torch.sqrt(y * y + z * z)
    ut = 0.5 * (1 + torch.tanh((0.5 - r) / (2 * (fp.theta + 0.01 * x))))
    env = torch.exp(-(r / 0.8) ** 2) * (r * r / (r * r + 0.1)) * torch.sin(math.pi / x.max() * x) ** 2
    M, g = fp.mach_j, fp.gamma
    T = (1 / fp.TR) * (1 - ut) + ut + 0.5 * (g - 1) * M * M * ut * (1 - ut)
    out = torch.empty((5, nk, nj, ni), dtype=torch.float64, device=DEV)
    out[0], out[1], out[4] = 1 / T, M * ut, 1 / g
    out[2], out[3] = 0, 0
    ti, tj, tk = (2 * math.pi * torch.arange(n, device=DEV, dtype=torch.float64) / n for n in (ni, nj, nk))
    for f, amp in enumerate((0.04, 0.1, 0.08, 0.08, 0.02)):
        scale = out[f].clone() if f in (0, 4) else 1.0
        for _ in range(3):
            m = rng.integers(1, 5, 3)
            ph = rng.uniform(0, 2 * math.pi, 3)
            w = (torch.sin(m[0] * ti + ph[0]).view(1, 1, ni) * torch.sin(m[1] * tj + ph[1]).view(1, nj, 1)
                 * torch.cos(m[2] * tk + ph[2]).view(nk, 1, 1))
            out[f] += amp * rng.uniform(0.3, 1.0) * scale * w * env
    return out.view(5, -1)


def _pinned(shape, like=None, dtype=torch.float64):
    t = torch.empty(shape, dtype=dtype, pin_memory=True)
    if like is not None:
        t.copy_(like)
    return t


def _dp(t):
    return ctypes.cast(t.data_ptr(), ctypes.POINTER(ctypes.c_double))


def _probe_points(spec):
    """The probe cylinder r = 3D of a jet box, 256 azimuths x 384 stations (fewer on a coarse grid)."""
    n_x = min(384, spec.dims[0])
    return I.cylinder_points(3.0, min(256, 4 * spec.dims[1]), n_x, 0.5, float(spec.x.max()) - 0.5)


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------

class _Out:
    """A program's buffers for the state it reads back: pinned FP64 as the library returns it, and the FP32 snapshot
    that an FP32 run keeps of it."""

    def __init__(self, n, prec):
        self.host = _pinned((5, n))
        self.snap = torch.empty((5, n), dtype=torch.float32) if prec != "fp64" else None

    def read(self, s, jet=0):
        les._check(s.h, les.lib().les_get_state_jet(s.h, jet, _dp(self.host), les.LES_STATE_CONSERVED))
        return self.host if self.snap is None else self.snap.copy_(self.host)


def prepare(case, seed):
    if case["do"] == "march":
        spec, fp = _spec(case), _flow(case, seed)
        s = les.Solver(spec, fp, PREC[case["prec"]])
        q = _pinned((5, spec.N), _jet_state(spec, fp, seed))
        les._check(s.h, les.lib().les_set_state_jet(s.h, 0, _dp(q), les.LES_STATE_PRIMITIVE))
        st = {"case": case, "solver": s, "out": _Out(spec.N, case["prec"])}
        if case["exchange"]:
            st["in"] = q
        if case["probe"]:
            xyz = _probe_points(spec)
            cap = max(1, case["steps"] // case["probe"])
            st["ring"] = torch.zeros((cap, 5, xyz.shape[1]), device=DEV,
                                     dtype=torch.float64 if case["prec"] == "fp64" else torch.float32)
            les.les_probe_surface(s.h, xyz, case["probe"], st["ring"].data_ptr(), cap)
        return st
    if case["do"] == "batch":
        jets = _batch(case["jets"], case["draw"])
        fps = [_batch_flow(f, seed) for _, f in jets]
        s = les.Solver([g for g, _ in jets], fps, PREC[case["prec"]])
        for j, ((g, _), f) in enumerate(zip(jets, fps)):
            q = _pinned((5, g.N), _jet_state(g, f, seed + j))
            les._check(s.h, les.lib().les_set_state_jet(s.h, j, _dp(q), les.LES_STATE_PRIMITIVE))
        return {"case": case, "solver": s, "outs": [_Out(g.N, case["prec"]) for g, _ in jets]}
    if case["do"] == "sums":
        qhat, rhs = _sums_in(case, seed)
        return {"case": case, "qhat": qhat, "rhs": rhs, "out": torch.empty(12, dtype=torch.float64, device=DEV)}
    return {"case": case, **_fwh_in(case, seed)}


@functools.lru_cache(maxsize=4)
def _batch(njets, draw_seed):
    return I.batch_jets(njets, seed=draw_seed)


def _batch_flow(f, seed):
    return I.FlowParams(**{**f.__dict__, "seed": f.seed + seed})


def _sums_in(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = case["points"]
    # cell volumes over two decades times a state, and a residual that is zero at a tenth of the points
    vol = torch.exp(4.6 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)) * 1e-4
    qhat = torch.randn((5, n), generator=g, device=DEV, dtype=torch.float64) * 0.1
    qhat[0] += 1.0
    qhat[4] += 2.0
    qhat *= vol
    rhs = torch.randn((5, n), generator=g, device=DEV, dtype=torch.float64) * 1e-3
    rhs *= (torch.rand(n, generator=g, device=DEV) > 0.1)
    return qhat, rhs


TR_FWH = 2.0


def _fwh_geometry(case):
    xyz, nrm, area = I.cylinder_panels(3.0, case["n_theta"], case["n_x"], 0.5, 29.5)
    obs = I.observer_arc(60.0, case["mics"], 15.0)
    c0, dtau = (1 / TR_FWH) ** 0.5, 0.1
    r = np.sqrt((obs ** 2).sum(0)[None, :] + (xyz ** 2).sum(0)[:, None] - 2 * xyz.T @ obs)
    t0 = float(r.max()) / c0 + 0.05
    dt_obs = dtau * case["dt_ratio"]
    # as many times as the frames cover
    nt = min(case["times"], int(((case["frames"] - 1) * dtau - 0.05 - t0 + float(r.min()) / c0) / dt_obs))
    return xyz, nrm, area, obs, c0, dtau, t0, dt_obs, nt


def _fwh_in(case, seed):
    """FP32 probe frames of four seeded monopoles on the jet axis radiating into the ambient."""
    xyz, nrm, area, obs, c0, dtau, t0, dt_obs, nt = _fwh_geometry(case)
    rng = np.random.default_rng(seed)
    sx, tc, amp = rng.uniform(3.0, 25.0, 4), rng.uniform(20.0, 60.0, 4), rng.uniform(0.05, 0.2, 4)
    P = torch.as_tensor(xyz, device=DEV)
    nfr, npts, sig, rho0, p0 = case["frames"], xyz.shape[1], 1.5, TR_FWH, 1 / 1.4
    ring = torch.empty((nfr, 5, npts), dtype=torch.float32, device=DEV)
    for m0 in range(0, nfr, 64):
        t = (torch.arange(m0, min(nfr, m0 + 64), device=DEV, dtype=torch.float64) * dtau)[:, None]
        p = torch.zeros((t.shape[0], npts), dtype=torch.float64, device=DEV)
        u = [torch.zeros_like(p) for _ in range(3)]
        for x_, t_, a_ in zip(sx, tc, amp):
            d = [P[0] - x_, P[1], P[2]]
            R = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
            tr = t - R / c0 - t_
            q = a_ * torch.exp(-(tr / sig) ** 2)
            qd = -2 * tr / sig ** 2 * q
            p += rho0 * qd / (4 * math.pi * R)
            ur = (qd / c0 + q / R) / (4 * math.pi * R) / R
            for c in range(3):
                u[c] += ur * d[c]
        o = ring[m0:m0 + t.shape[0]]
        o[:, 0], o[:, 4] = (rho0 + p / c0 ** 2).float(), (p0 + p).float()
        for c in range(3):
            o[:, 1 + c] = u[c].float()
    return {"ring": ring, "args": (xyz, nrm, area, dtau, p0, c0, obs, t0, dt_obs, nt)}


def run(state):
    c = state["case"]
    if c["do"] == "sums":
        les.les_diag_sums_noalloc(state["qhat"].data_ptr(), state["rhs"].data_ptr(), c["points"],
                                  state["out"].data_ptr())
        return state["out"]
    if c["do"] == "fwh":
        p = les.les_fwh(state["ring"].data_ptr(), les.LES_FP32, c["frames"], c["frames"], *state["args"])
        return p.astype(np.float32)  # the signal, kept in the precision of the frames it came from
    s = state["solver"]
    if c["do"] == "batch":
        s.step(c["steps"])
        return [o.read(s, j) for j, o in enumerate(state["outs"])]
    if c["exchange"]:
        les._check(s.h, les.lib().les_set_state_jet(s.h, 0, _dp(state["in"]), les.LES_STATE_PRIMITIVE))
    res = {}
    if c["monitor"]:
        watch = []
        for k in range(c["monitor"], c["steps"] + 1, c["monitor"]):
            s.step(c["monitor"])
            d = s.diagnostics(check=False)
            watch.append([d["max_abs_rhs_rho"], *d["l2_rhs"], *d["sum_qhat"]])
        res["monitor"] = np.array(watch, dtype=np.float32)
        s.step(c["steps"] % c["monitor"])
    else:
        s.step(c["steps"])
    res["state"] = state["out"].read(s)
    if c["probe"]:
        res["probe"] = state["ring"]
    return res


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------

def _march_work(mesh, n, prec, steps):
    # per point and stage: Q(l-1) and Q(0) in (the first stage reads Q(0) alone), Q(l) out: 14 values on average; a
    # curvilinear mesh also reads nine cofactors and the Jacobian, a product grid only 1-D spacings
    es = 8 if prec == "fp64" else 4
    vals = 24 if mesh == "polar" else 14
    # each point quantity and each interface flux once: 706 operations with general metrics, about 400 with
    # diagonal ones
    flops = 706 if mesh == "polar" else 400
    return {"bytes": steps * 5.0 * n * vals * es + 5.0 * n * 8, "flops": steps * 5.0 * n * flops}


def work(case):
    if case["do"] == "sums":
        return {"bytes": 80.0 * case["points"] + 96, "flops": 50.0 * case["points"]}
    if case["do"] == "fwh":
        nt = _fwh_geometry(case)[-1]
        npts = case["n_theta"] * case["n_x"]
        return {"bytes": 20.0 * npts * case["frames"] + 56.0 * npts + 8.0 * case["mics"] * nt,
                "flops": 42.0 * npts * case["mics"] * nt + 40.0 * npts * case["frames"]}
    if case["do"] == "batch":
        w = [_march_work("jet", g.N, case["prec"], case["steps"]) for g, _ in _batch(case["jets"], case["draw"])]
        return {k: sum(v[k] for v in w) for k in ("bytes", "flops")}
    n = case["ni"] * case["nj"] * case["nk"]
    return _march_work(case["mesh"], n, case["prec"], case["steps"])


# ---------------------------------------------------------------------------
# exact: the method stated in 64-bit torch
# ---------------------------------------------------------------------------

def _sl(a, s):
    """Index of an array [..., k, j, i] along grid axis a (0 = i)."""
    return (Ellipsis,) + (s,) + (slice(None),) * a


def _splitmix(seed, n):
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (n + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


class _Jet:
    """The filtered Navier-Stokes stage, its boundary conditions and time step on one grid (arrays [k, j, i])."""

    def __init__(self, spec, fp):
        self.fp, self.bc, self.per = fp, spec.bc, spec.periodic
        self.n = spec.dims
        ni, nj, nk = spec.dims
        X = [torch.as_tensor(v, device=DEV).view(nk, nj, ni) for v in (spec.x, spec.y, spec.z)]
        D = self.D
        self.m = [[None] * 3 for _ in range(3)]
        for a in range(3):
            b, d = (a + 1) % 3, (a + 2) % 3
            for c in range(3):
                c1, c2 = (c + 1) % 3, (c + 2) % 3
                self.m[a][c] = D(X[c1] * D(X[c2], d), b) - D(X[c1] * D(X[c2], b), d)
        t = [[D(X[c], a) for a in range(3)] for c in range(3)]
        self.jinv = (t[0][0] * (t[1][1] * t[2][2] - t[1][2] * t[2][1])
                     - t[0][1] * (t[1][0] * t[2][2] - t[1][2] * t[2][0])
                     + t[0][2] * (t[1][0] * t[2][1] - t[1][1] * t[2][0]))
        if not any(self.per):  # a product grid's cross terms are zeros; keep them out of the sums
            for a in range(3):
                for c in range(3):
                    if a != c:
                        self.m[a][c] = None
        self.rj = 1 / torch.where(self.jinv > 0, self.jinv, torch.ones_like(self.jinv))
        self.ut = 0.5 * (1 + torch.tanh((0.5 - torch.sqrt(X[1][:, :, 0] ** 2 + X[2][:, :, 0] ** 2)) / (2 * fp.theta)))

    def D(self, f, a):
        if self.per[a]:
            return 0.5 * (torch.roll(f, -1, -1 - a) - torch.roll(f, 1, -1 - a))
        o = torch.empty_like(f)
        s = lambda k: f[_sl(a, k)]  # noqa: E731
        o[_sl(a, slice(1, -1))] = 0.5 * (s(slice(2, None)) - s(slice(0, -2)))
        o[_sl(a, 0)] = -1.5 * s(0) + 2 * s(1) - 0.5 * s(2)
        o[_sl(a, -1)] = 1.5 * s(-1) - 2 * s(-2) + 0.5 * s(-3)
        return o

    def dot(self, a, v):
        """m_a . v over the cofactors that are there."""
        s = None
        for c in range(3):
            if self.m[a][c] is not None:
                s = self.m[a][c] * v[c] if s is None else s + self.m[a][c] * v[c]
        return s

    def prim(self, Q):
        rho = Q[0]
        u = [Q[1 + c] / rho for c in range(3)]
        p = (self.fp.gamma - 1) * (Q[4] - 0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2))
        return rho, u, p, self.fp.gamma * p / rho

    def lam(self, u, T):
        out = []
        for a in range(3):
            nrm = sum(self.m[a][c] ** 2 for c in range(3) if self.m[a][c] is not None).sqrt()
            out.append(((self.dot(a, u)).abs() + T.sqrt() * nrm) * self.rj)
        return out

    def dt(self, Q):
        rho, u, p, T = self.prim(Q)
        return self.fp.cfl / float(sum(self.lam(u, T)).max())

    def rhs(self, Q):
        fp, g = self.fp, self.fp.gamma
        rho, u, p, T = self.prim(Q)
        S = fp.S1_dim / (fp.TR * fp.T_inf_dim)
        mu = T.sqrt() * T * (1 + S) / (T + S)
        rH = Q[4] + p
        W = [Q[0], Q[1], Q[2], Q[3], rH]
        lam = self.lam(u, T)
        lb = [lam[a] + (lam[a] * lam[(a + 1) % 3]).sqrt() + (lam[a] * lam[(a + 2) % 3]).sqrt() for a in range(3)]
        phi = [*u, T]
        d = [[self.D(f, a) for a in range(3)] for f in phi]
        gr = [[sum(self.m[b][c] * d[i][b] for b in range(3) if self.m[b][c] is not None) * self.rj for c in range(3)]
              for i in range(3)]
        ss = sum(2 * gr[i][i] ** 2 for i in range(3))
        for i, j in ((0, 1), (0, 2), (1, 2)):
            ss = ss + (gr[i][j] + gr[j][i]) ** 2
        mus = rho * (fp.Cs * self.jinv.clamp(min=0) ** (1 / 3)) ** 2 * ss.sqrt()
        del gr, ss
        mue = mu / fp.Re + mus
        kap = (mu / (fp.Re * fp.Pr) + mus / fp.Pr_sgs) / (g - 1)
        R = torch.zeros_like(Q)
        for a in range(3):
            per, ax = self.per[a], -1 - a
            if per:
                L = lambda f: f  # noqa: E731
                Rt = lambda f: torch.roll(f, -1, ax)  # noqa: E731
            else:
                L = lambda f: f[_sl(a, slice(0, -1))]  # noqa: E731
                Rt = lambda f: f[_sl(a, slice(1, None))]  # noqa: E731
            avg = lambda f: 0.5 * (L(f) + Rt(f))  # noqa: E731
            # sensor
            if per:
                pm, pp = torch.roll(p, 1, ax), torch.roll(p, -1, ax)
                nu = (pp - 2 * p + pm).abs() / (pp + 2 * p + pm)
            else:
                pm, pc, pp = (p[_sl(a, s)] for s in (slice(0, -2), slice(1, -1), slice(2, None)))
                v = (pp - 2 * pc + pm).abs() / (pp + 2 * pc + pm)
                nu = torch.cat([v[_sl(a, slice(0, 1))], v, v[_sl(a, slice(-1, None))]], ax)
            eps2 = fp.k2 * torch.maximum(L(nu), Rt(nu))
            eps4 = (fp.k4 - eps2).clamp(min=0)
            jb = avg(self.jinv)
            rjb = torch.where(jb > 0, 1 / jb, torch.zeros_like(jb))
            sc = jb * avg(lb[a])
            # centred flux and dissipation
            JU = self.dot(a, u)
            H = []
            for f in range(5):
                F = W[f] * JU
                if 1 <= f <= 3 and self.m[a][f - 1] is not None:
                    F = F + p * self.m[a][f - 1]
                dW = Rt(W[f]) - L(W[f])
                if per:
                    dm, dp = torch.roll(dW, 1, ax), torch.roll(dW, -1, ax)
                else:
                    dm = torch.cat([-dW[_sl(a, slice(0, 1))], dW[_sl(a, slice(0, -1))]], ax)
                    dp = torch.cat([dW[_sl(a, slice(1, None))], -dW[_sl(a, slice(-1, None))]], ax)
                H.append(avg(F) - sc * (eps2 * dW - eps4 * (dp - 2 * dW + dm)))
            # compact viscous flux
            A = [[None if self.m[b][c] is None else avg(self.m[b][c]) * rjb for c in range(3)] for b in range(3)]
            dd = [[Rt(f) - L(f) if b == a else avg(d[i][b]) for b in range(3)] for i, f in enumerate(phi)]
            G = [[sum(A[b][c] * dd[i][b] for b in range(3) if A[b][c] is not None) for c in range(3)]
                 for i in range(4)]
            div = G[0][0] + G[1][1] + G[2][2]
            mub, kb = avg(mue) * jb, avg(kap) * jb
            for i in range(3):
                s = None
                for c in range(3):
                    if A[a][c] is None:
                        continue
                    tau = G[i][c] + G[c][i]
                    if i == c:
                        tau = tau - (2 / 3) * div
                    s = A[a][c] * tau if s is None else s + A[a][c] * tau
                s = mub * s
                H[1 + i] = H[1 + i] - s
                H[4] = H[4] - s * avg(u[i])
            for c in range(3):
                if A[a][c] is not None:
                    H[4] = H[4] - kb * A[a][c] * G[3][c]
            for f in range(5):
                if per:
                    R[f] += H[f] - torch.roll(H[f], 1, ax)
                else:
                    R[f][_sl(a, slice(1, -1))] += H[f][_sl(a, slice(1, None))] - H[f][_sl(a, slice(0, -1))]
        for a in range(3):
            if not self.per[a]:
                R[_sl(a, 0)] = 0
                R[_sl(a, -1)] = 0
        return R

    def cons(self, rho, u, p):
        return torch.stack([rho, rho * u[0], rho * u[1], rho * u[2],
                            p / (self.fp.gamma - 1) + 0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)])

    def farfield(self, Qe, nrm):
        g, TR = self.fp.gamma, self.fp.TR
        rho, u, p, T = self.prim(Qe)
        ce, cinf = T.sqrt(), math.sqrt(1 / TR)
        qn = u[0] * nrm[0] + u[1] * nrm[1] + u[2] * nrm[2]
        rp, rm = qn + 2 * ce / (g - 1), -2 * cinf / (g - 1)
        qf, cf = 0.5 * (rp + rm), 0.25 * (g - 1) * (rp - rm)
        mn = qn / ce
        ro = (rho ** g * cf * cf / (g * p)) ** (1 / (g - 1))
        ri = (TR ** g * cf * cf) ** (1 / (g - 1))
        out = self.cons(ro, [u[c] + (qf - qn) * nrm[c] for c in range(3)], ro * cf * cf / g)
        inn = self.cons(ri, [qf * nrm[c] for c in range(3)], ri * cf * cf / g)
        amb = self.cons(torch.full_like(rho, TR), [torch.zeros_like(rho)] * 3, torch.full_like(rho, 1 / g))
        return torch.where(mn >= 1, Qe, torch.where(mn <= -1, amb, torch.where(mn >= -1e-8, out, inn)))

    def exit(self, Qe, nrm):
        g = self.fp.gamma
        rho, u, p, T = self.prim(Qe)
        mn = (u[0] * nrm[0] + u[1] * nrm[1] + u[2] * nrm[2]) / T.sqrt()
        ei = p / ((g - 1) * rho)
        r = 1 / (g * (g - 1) * ei)
        Qf = torch.stack([r, r * u[0], r * u[1], r * u[2], r * (ei + 0.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2))])
        return torch.where(mn >= 1, Qe, Qf)

    def inflow(self, Qe, nrm, level):
        fp = self.fp
        g, M, ut = fp.gamma, fp.mach_j, self.ut
        far = self.farfield(Qe, nrm)
        T = (1 / fp.TR) * (1 - ut) + ut + 0.5 * (g - 1) * M * M * ut * (1 - ut)
        u = [M * ut, torch.zeros_like(ut), torch.zeros_like(ut)]
        if level > 0:
            nk, nj = ut.shape
            base = (level - 1) * nk * nj * 3
            h = _splitmix(fp.seed, np.arange(nk * nj * 3, dtype=np.uint64) + np.uint64(base))
            h = (h >> np.uint64(11)).astype(np.float64) / 9007199254740992.0
            w = torch.as_tensor(fp.noise_amp * M * (2 * h - 1), device=DEV).view(nk, nj, 3)
            u = [u[c] + w[:, :, c] for c in range(3)]
        jet = self.cons(1 / T, u, torch.full_like(ut, 1 / g))
        return torch.where(ut < 0.01, far, jet)

    def faces(self, Q, level):
        """Boundary conditions of a time level, faces y, z, x in turn."""
        for a in (1, 2, 0):
            if a == 1 and self.bc[2] == I.BC_CENTERLINE:
                Q[:, :, 0, :] = Q[:, :, 1, :].mean(1, keepdim=True)
            if self.per[a]:
                continue
            for side in (0, 1):
                kind = self.bc[2 * a + side]
                if kind == I.BC_CENTERLINE:
                    continue
                at, inner = (-1, -2) if side else (0, 1)
                v = [torch.zeros_like(self.jinv[_sl(a, at)]) if self.m[a][c] is None
                     else (1 if side else -1) * self.m[a][c][_sl(a, at)] for c in range(3)]
                r = torch.sqrt(v[0] ** 2 + v[1] ** 2 + v[2] ** 2)
                nrm = [x / r for x in v]
                Qe = Q[_sl(a, inner)]
                if kind == I.BC_FARFIELD:
                    Q[_sl(a, at)] = self.farfield(Qe, nrm)
                elif kind == I.BC_EXIT:
                    Q[_sl(a, at)] = self.exit(Qe, nrm)
                else:
                    Q[_sl(a, at)] = self.inflow(Qe, nrm, level)
        return Q

    def step(self, Q, level, dt):
        Q0 = Q
        for al in ALPHA:
            Q = Q0 - (al * dt) * self.rhs(Q) * self.rj
            Q = self.faces(Q, level + 1)
        return Q


def _start(spec, fp, seed):
    jet = _Jet(spec, fp)
    ni, nj, nk = spec.dims
    w = _jet_state(spec, fp, seed).view(5, nk, nj, ni)
    Q = jet.faces(jet.cons(w[0], [w[1], w[2], w[3]], w[4]), 0)
    return jet, Q, jet.dt(Q)


def _probe_exact(spec, fp, Q, xyz):
    """Trilinear values of the primitives of Q at the points."""
    ni, nj, nk = spec.dims
    ax = (spec.x[:ni], spec.y.reshape(nk, nj, ni)[0, :, 0], spec.z.reshape(nk, nj, ni)[:, 0, 0])
    lo, w = [], []
    for a in range(3):
        k = np.clip(np.searchsorted(ax[a], xyz[a]) - 1, 0, len(ax[a]) - 2)
        lo.append(torch.as_tensor(k, device=DEV))
        w.append(torch.as_tensor((xyz[a] - ax[a][k]) / (ax[a][k + 1] - ax[a][k]), device=DEV))
    out = 0
    for c in range(8):
        up = [(c >> a) & 1 for a in range(3)]
        q = Q[:, lo[2] + up[2], lo[1] + up[1], lo[0] + up[0]]
        u = q[1:4] / q[0]
        p = (fp.gamma - 1) * (q[4] - 0.5 * q[0] * (u ** 2).sum(0))
        wt = 1.0
        for a in range(3):
            wt = wt * (w[a] if up[a] else 1 - w[a])
        out = out + wt * torch.cat([q[:1], u, p[None]])
    return out


def _march_exact(case, seed):
    spec, fp = _spec(case), _flow(case, seed)
    jet, Q, dt = _start(spec, fp, seed)
    res, watch, frames = {}, [], []
    xyz = _probe_points(spec) if case["probe"] else None
    for n in range(case["steps"]):
        Q = jet.step(Q, n, dt)
        if case["monitor"] and (n + 1) % case["monitor"] == 0:
            R = jet.rhs(Q)
            s = torch.where(jet.jinv > 0, jet.jinv, torch.ones_like(jet.jinv))
            watch.append([float(R[0].abs().max()), *[float(R[f].square().sum().sqrt()) for f in range(5)],
                          *[float((s * Q[f]).sum()) for f in range(5)]])
        if case["probe"] and (n + 1) % case["probe"] == 0:
            frames.append(_probe_exact(spec, fp, Q, xyz))
    if case["monitor"]:
        res["monitor"] = np.array(watch)
    res["state"] = Q.reshape(5, -1)
    if case["probe"]:
        cap = max(1, case["steps"] // case["probe"])
        ring = torch.zeros((cap, *frames[0].shape), dtype=torch.float64, device=DEV)
        for f, v in enumerate(frames):
            ring[f % cap] = v
        res["probe"] = ring
    return res


def _fwh_exact(case, seed):
    st = _fwh_in(case, seed)
    xyz, nrm, area, dtau, p0, c0, obs, t0, dt_obs, nt = st["args"]
    ring, N = st["ring"], case["frames"]
    out = torch.zeros((case["mics"], nt), dtype=torch.float64, device=DEV)
    t = t0 + dt_obs * torch.arange(nt, dtype=torch.float64, device=DEV)
    for j0 in range(0, xyz.shape[1], 8192):
        sl = slice(j0, min(xyz.shape[1], j0 + 8192))
        w = ring[:, :, sl].double()
        n = torch.as_tensor(nrm[:, sl], device=DEV)
        un = (w[:, 1:4] * n).sum(1)
        V = torch.cat([(w[:, 4:5] - p0) * n + w[:, 0:1] * w[:, 1:4] * un[:, None], (w[:, 0] * un)[:, None]], 1)
        dV = torch.empty_like(V)
        dV[1:-1] = (V[2:] - V[:-2]) / (2 * dtau)
        dV[0] = (-3 * V[0] + 4 * V[1] - V[2]) / (2 * dtau)
        dV[-1] = (3 * V[-1] - 4 * V[-2] + V[-3]) / (2 * dtau)
        P, A = torch.as_tensor(xyz[:, sl], device=DEV), torch.as_tensor(area[sl], device=DEV)
        for o in range(case["mics"]):
            d = [float(obs[c, o]) - P[c] for c in range(3)]
            r = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
            Lr = sum(V[:, c] * d[c] for c in range(3)) / r
            dLr = sum(dV[:, c] * d[c] for c in range(3)) / r
            E = (A / (4 * math.pi) * (dV[:, 3] / r + dLr / (c0 * r) + Lr / r ** 2)).T.contiguous()
            s = (t[None, :] - (r / c0)[:, None]) / dtau
            m = s.floor().clamp(0, N - 2).long()
            a = E.gather(1, m)
            out[o] += (a + (s - m) * (E.gather(1, m + 1) - a)).sum(0)
    return out


def exact(case, seed):
    if case["do"] == "sums":
        q, r = _sums_in(case, seed)
        return torch.cat([r[0].abs().max()[None], r.square().sum(1).sqrt(), q.sum(1),
                          torch.zeros(1, dtype=torch.float64, device=DEV)])
    if case["do"] == "fwh":
        return _fwh_exact(case, seed)
    if case["do"] == "batch":
        outs = []
        for j, (g, f) in enumerate(_batch(case["jets"], case["draw"])):
            jet, Q, dt = _start(g, _batch_flow(f, seed), seed + j)
            for n in range(case["steps"]):
                Q = jet.step(Q, n, dt)
            outs.append(Q.reshape(5, -1))
        return outs
    return _march_exact(case, seed)
