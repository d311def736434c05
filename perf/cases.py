"""Timed cases of the FTH-MS library: the calls a program makes through the C ABI binding, over the range of
sizes, precisions and options that the workloads use.

Three kinds of case:
  bessel         fthms_bessel0 on device arrays
  self, noalloc  one arc's Nystrom matrix (fthms_assemble_self, fthms_assemble_self_noalloc)
  job            a whole prepared job: run, wait, output traces, every arc's summed densities on the device
  served         a burst of requests through the request server: submit, wait, traces, release

A job's geometry is one of the workloads' families: "small" (a few arcs, tiny sizes), "disk" (interior point
source), "obstacles" (exterior, plane wave), "cavity" (12-arc star, several windows), "arcs" (open and closed
elliptic arcs, fixed N).  The seed moves obstacles, phases, sources and carriers; sizes come from the case.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import workloads as wl
from paper_2507_05725_gb300 import fthms as F

_DEVICE = "cuda"


# ---------------------------------------------------------------------------------------------
# The cases

def _job(name, geometry, **kw):
    case = {"name": name, "kind": "job", "geometry": geometry, "precision": 0, "cross_mode": 0, "graph": False,
            "sampled": False, "shapes": ""}
    case.update(kw)
    return case


def listed():
    return [
        # the kernel-level entry points: special functions on a device array, and one arc's matrix for callers
        # that bring their own solver (a small latency-bound one without allocation, and a large one)
        {"name": "bessel0-1e6", "kind": "bessel", "n": 1000003},
        {"name": "noalloc-N96", "kind": "noalloc", "N": 96, "kappa": 24.0},
        {"name": "self-N777", "kind": "self", "N": 777, "kappa": 180.0},
        # the smallest jobs: a quick look at a geometry, where launches and host latency count
        _job("small-fp64", "small", W=10.0, L=33, M=2, Q=1, arcs=3, curves=1, shape=3),
        # an interior problem driven by a point source, checked against its exact field (first configuration)
        _job("disk3-fp64", "disk", W=24.0, L=257, M=8, Q=1, arcs=3, N=96),
        # an exterior scattering problem with the wavelength rule (second configuration): the FP64 form, and the
        # mixed form replayed as a graph by a program that runs one job again and again
        _job("obstacles-fp64", "obstacles", W=60.0, L=1025, M=12, Q=1),
        _job("obstacles-mixed-graph", "obstacles", W=60.0, L=1025, M=12, Q=1, precision=1, graph=True),
        # the same family driven by measured samples of a signal, FP64-kept mixed form, shorter band
        _job("obstacles-sampled", "obstacles", W=30.0, L=321, M=5, Q=1, precision=2, sampled=True),
        # high-frequency arcs with fixed N in the FP64-kept mixed form with tuned shapes: cross rows stored, and
        # (N = 1024) evaluated every step
        _job("arcs-N512", "arcs", W=300.0, L=385, M=8, Q=2, N=512, precision=2, shapes="1,256,512,256,256"),
        _job("arcs-N1024", "arcs", W=300.0, L=385, M=3, Q=2, N=1024, precision=2, cross_mode=1),
        # the many-arc cavity with four time windows, cross rows evaluated every step
        _job("cavity12-Q4", "cavity", W=60.0, L=257, M=5, Q=4, arcs=12, precision=1, cross_mode=1),
        # a burst of requests of different geometries and bands arriving at a server
        {"name": "served-8", "kind": "served", "requests": 8, "wmin": 20.0, "wmax": 60.0, "L": 257, "arcs_max": 6,
         "precision": 1, "inflight": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# the most a drawn job may cost: the flops of the largest listed one
_MOST_FLOPS = 4.0e12


def draw(rng):
    while True:
        case = _draw(rng)
        if case["kind"] != "job":
            return case
        w = work(case)
        if w["flops"] <= _MOST_FLOPS and _device_gb(case) <= 60.0:
            return case


def _draw(rng):
    kind = rng.choice(["bessel", "noalloc", "self", "small", "disk", "disk", "obstacles", "obstacles", "obstacles",
                       "arcs", "arcs", "cavity", "served"])
    if kind == "bessel":
        return {"kind": "bessel", "n": _log_int(rng, 1000, 4000000)}
    if kind in ("noalloc", "self"):
        return {"kind": kind, "N": _log_int(rng, 8, 256 if kind == "noalloc" else 1024),
                "kappa": round(math.exp(rng.uniform(math.log(0.5), math.log(300.0))), 3)}
    if kind == "served":
        return {"kind": "served", "requests": rng.randint(2, 8), "wmin": 20.0, "wmax": rng.choice([40.0, 60.0]),
                "L": rng.choice([129, 257]), "arcs_max": rng.randint(4, 8), "precision": rng.choice([0, 1, 2]),
                "inflight": rng.choice([1, 2, 4])}
    if kind == "small":
        c = _job("", "small", W=round(rng.uniform(6.0, 12.0), 2), L=rng.choice([33, 49, 65]), M=rng.randint(2, 4),
                 Q=rng.choice([1, 1, 2]), arcs=rng.choice([2, 3, 4, 5]), curves=rng.choice([1, 2]),
                 shape=rng.randint(0, 99), precision=rng.choice([0, 1, 2]))
    elif kind == "disk":
        c = _job("", "disk", W=24.0, L=rng.choice([193, 257, 301]), M=rng.randint(3, 8), Q=rng.choice([1, 2]),
                 arcs=rng.choice([3, 4, 5]), N=_log_int(rng, 64, 200), precision=rng.choice([0, 0, 1, 2]),
                 cross_mode=rng.choice([0, 0, 1]))
    elif kind == "obstacles":
        W = round(math.exp(rng.uniform(math.log(16.0), math.log(60.0))), 2)
        L = _log_int(rng, 257, 1025)
        c = _job("", "obstacles", W=W, L=L, M=rng.randint(3, 12), Q=rng.choice([1, 1, 2]),
                 precision=rng.choice([0, 1, 2]), graph=rng.random() < 0.3, sampled=rng.random() < 0.3,
                 cross_mode=rng.choice([0, 0, 0, 1]))
    elif kind == "arcs":
        c = _job("", "arcs", W=300.0, L=rng.choice([385, 389]), M=rng.randint(2, 8), Q=rng.choice([1, 2]),
                 N=_log_int(rng, 480, 1100), precision=2, cross_mode=rng.choice([0, 1]),
                 shapes=rng.choice(["", "1,256,512,256,256"]))
    else:
        W = round(rng.uniform(30.0, 60.0), 2)
        c = _job("", "cavity", W=W, L=rng.choice([257, 273, 301]), M=rng.randint(2, 5), Q=rng.choice([2, 3, 4]),
                 arcs=rng.choice([6, 8, 12]), precision=rng.choice([1, 2]), cross_mode=1)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------
# Problems

def _problem(case, seed):
    g = case["geometry"]
    rng = np.random.default_rng([7, int(seed) & 0x7FFFFFFF])
    if g == "small":
        # the shape comes with the case (it sets the node counts), its place and the signal with the seed
        p = wl.random_small(case["shape"], n_arcs_per_curve=case["arcs"], n_curves=case["curves"], L=case["L"],
                            M=case["M"], Q=case["Q"], W=case["W"])
        p["signal"].update(carrier=float(rng.uniform(3.0, 6.0)), centre=float(rng.uniform(2.2, 2.8)),
                           z0=[4.0 * (case["curves"] - 1) + float(rng.uniform(2.0, 2.6)), float(rng.uniform(-1, 1))])
    elif g == "disk":
        p = wl.config1(L=case["L"], M=case["M"], N=case["N"])
        p["arcs"] = wl.split_closed_curve(0, case["arcs"], 1.25, float(rng.uniform(0.0, 2.0 * math.pi)))
        a, r = float(rng.uniform(0.0, 2.0 * math.pi)), float(rng.uniform(1.9, 2.3))
        p["signal"].update(z0=[r * math.cos(a), r * math.sin(a)], carrier=float(rng.uniform(3.6, 4.4)))
        period = 2.0 * math.pi * (case["L"] - 1) / case["W"]
        p["options"].update(W=case["W"], Q=case["Q"], H=min(20.0, 0.45 * period))
    elif g == "obstacles":
        period = 2.0 * math.pi * (case["L"] - 1) / case["W"]
        big = case["W"] > 30.0
        p = wl.config2(seed=int(seed) & 0x7FFFFFFF, L=case["L"], M=case["M"], W=case["W"], Q=case["Q"],
                       H=min(40.0, 0.45 * period), n_period=4096 if big else 2048)
        if case["sampled"]:
            p = wl.with_samples(p, wl.multipulse_samples(t_lag=float(rng.uniform(1.5, 2.5)), pulses=3))
        else:
            p["signal"]["carrier"] = min(10.0, 0.5 * case["W"]) * float(rng.uniform(0.9, 1.1))
    elif g == "arcs":
        p = wl.config4(N=case["N"], seed=int(seed) & 0x7FFFFFFF, L=case["L"], M=case["M"], W=case["W"], Q=case["Q"],
                       cross_mode=case["cross_mode"])
    elif g == "cavity":
        p = wl.config3(seed=int(seed) & 0x7FFFFFFF, L=case["L"], M=case["M"], W=case["W"], Q=case["Q"], n_period=2048,
                       carrier=0.4 * case["W"] * float(rng.uniform(0.9, 1.1)), centre=12.0, width=3.0)
        # the arcs turn with the star, so that their lengths (and node counts) are the same for every seed
        phase = math.atan2(-p["curves"][0]["bx"][6], p["curves"][0]["ax"][6])
        p["arcs"] = wl.split_closed_curve(0, case["arcs"], 1.25, -phase / 5.0)
    else:
        raise ValueError(g)
    o = p["options"]
    o["cross_mode"] = case["cross_mode"]
    if case["precision"] > 0:
        o["refine_max"] = 8
    if case["shapes"]:
        o["shapes"] = tuple(int(v) for v in case["shapes"].split(","))
    return p


def _requests(case, seed):
    return wl.served_requests(int(seed) & 0x7FFFFFFF, case["requests"], wmax=(case["wmin"], case["wmax"]),
                              Ls=(case["L"],), arcs=(2, case["arcs_max"]))


def _arc_curve(rng):
    """A curve and an arc of it for the single-matrix calls."""
    curve = wl.star(0.3, 5, float(rng.uniform(0.0, 2.0 * math.pi)))
    c = float(rng.uniform(0.0, 2.0 * math.pi))
    return curve, (c - 0.9, c + 0.9)


# ---------------------------------------------------------------------------------------------
# State and pass

_CTX = {}


def _context():
    """One context for the program, on a stream that its torch code can wait for."""
    if "ctx" not in _CTX:
        torch.cuda.init()
        _CTX["stream"] = torch.cuda.Stream()
        _CTX["ctx"] = F.fthms_create(torch.cuda.current_device(), 0, _CTX["stream"].cuda_stream)
    return _CTX["ctx"], _CTX["stream"]


def _bessel_input(case, seed):
    g = torch.Generator(device="cpu").manual_seed(int(seed))
    u = torch.rand(case["n"], generator=g, dtype=torch.float64)
    # kernel arguments kappa R: from the near diagonal of a low frequency to the far field of a high one
    return torch.exp(math.log(1e-3) + u * (math.log(2000.0) - math.log(1e-3)))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "bessel":
        z = _bessel_input(case, seed).to(_DEVICE)
        return {"kind": kind, "z": z, "out": [torch.empty_like(z) for _ in range(3)]}
    if kind in ("self", "noalloc"):
        curve, arc = _arc_curve(np.random.default_rng([11, int(seed) & 0x7FFFFFFF]))
        return {"kind": kind, "curve": curve, "arc": arc, "N": case["N"], "kappa": case["kappa"],
                "A": torch.empty((case["N"], case["N"]), dtype=torch.complex128, device=_DEVICE)}
    if kind == "served":
        server = _CTX.get(("server", case["inflight"]))
        if server is None:
            torch.cuda.init()
            server = F.Server(torch.cuda.current_device(), 0, case["inflight"])
            _CTX[("server", case["inflight"])] = server
        return {"kind": kind, "server": server, "problems": _requests(case, seed), "precision": case["precision"]}
    ctx, stream = _context()
    problem = _problem(case, seed)
    job = F.Job(ctx, problem, keep_densities=False, precision=case["precision"])
    if case["graph"]:
        F.fthms_use_graph(job.req, True)
    counts = job.node_counts().sum(axis=1)
    dens = [[torch.empty(int(n), dtype=torch.complex128, device=_DEVICE) for _ in range(job.Q)] for n in counts]
    return {"kind": kind, "job": job, "stream": stream, "dens": dens}


def run(state):
    kind = state["kind"]
    if kind == "bessel":
        z, (j0, y0, yh) = state["z"], state["out"]
        F.fthms_bessel0(z.data_ptr(), j0.data_ptr(), y0.data_ptr(), yh.data_ptr(), z.numel(),
                        torch.cuda.current_stream().cuda_stream)
        return {"j0": j0, "y0": y0, "yhat0": yh}
    if kind in ("self", "noalloc"):
        f = F.fthms_assemble_self if kind == "self" else F.fthms_assemble_self_noalloc
        f(state["curve"], state["arc"], state["N"], state["kappa"], state["A"].data_ptr(),
          torch.cuda.current_stream().cuda_stream)
        return state["A"]
    if kind == "served":
        s = state["server"]
        tickets = [s.submit(p, precision=state["precision"]) for p in state["problems"]]
        out = []
        for t in tickets:
            s.wait(t)
            out.append(s.traces(t))
            s.release(t)
        return out
    job = state["job"]
    job.run().wait()
    traces = job.traces()
    for j, row in enumerate(state["dens"]):
        for q, d in enumerate(row):
            F.fthms_densities_dev(job.req, j, 0, q, d.data_ptr(), 2 * d.numel())
    torch.cuda.current_stream().wait_stream(state["stream"])
    if job.Q * job.P > 40:          # one array per arc
        return {"traces": traces, "densities": [torch.cat(row) for row in state["dens"]]}
    return {"traces": traces, "densities": state["dens"]}


# ---------------------------------------------------------------------------------------------
# Work

def _sizes(p):
    """Node counts [P, L-1], transfer-mesh rows per receiving arc, of a problem."""
    o = p["options"]
    arcs = [_Arc(p["curves"][c], c, a, b) for c, a, b in p["arcs"]]
    om = np.arange(1, o["L"]) * (o["W"] / (o["L"] - 1))
    N = np.stack([_node_counts(o, a.length(), om) for a in arcs]) if arcs else np.zeros((0, 0))
    return arcs, N


def _job_work(p):
    """LU, triangular solves, cross-arc and observation matvecs; outputs written once."""
    o = p["options"]
    arcs, N = _sizes(p)
    N = N.astype(np.float64)
    P, M, Q = len(arcs), o["M"], o["Q"]
    nmax = N[:, -1]
    n_obs = len(o["obs"])
    on_curve = {}
    for a in arcs:
        on_curve[a.ci] = on_curve.get(a.ci, 0) + 1
    entries = 0.0
    for j, a in enumerate(arcs):
        rows = n_obs
        for k, b in enumerate(arcs):
            if k != j:
                rows += nmax[k] * (0.9 if on_curve[b.ci] > 1 else 1.0)
        entries += rows * N[j].sum()
    flops = (8.0 / 3.0) * (N ** 3).sum() + 8.0 * Q * M * ((N ** 2).sum() + entries)
    return {"bytes": 16.0 * Q * N.sum() + 8.0 * n_obs * o["n_tout"], "flops": float(flops)}


def _device_gb(case):
    p = _problem(case, 1)
    return F.fthms_plan_info(F.Marshalled(p, keep_densities=False, precision=case["precision"]))[0] / 1e9


def work(case):
    kind = case["kind"]
    if kind == "bessel":
        return {"bytes": 32.0 * case["n"], "flops": 50.0 * case["n"]}
    if kind in ("self", "noalloc"):
        n = case["N"]
        return {"bytes": 16.0 * n * n, "flops": 50.0 * n * (n + 1) / 2}
    if kind == "served":
        ws = [_job_work(p) for p in _requests(case, 1)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    return _job_work(_problem(case, 1))


# ---------------------------------------------------------------------------------------------
# The same results in plain torch and numpy, 64 bits

def exact(case, seed):
    kind = case["kind"]
    if kind == "bessel":
        z = _bessel_input(case, seed)
        j0, y0 = _bessel0(z)
        yh = y0 - (2.0 / math.pi) * (torch.log(0.5 * z) + np.euler_gamma) * j0
        return {"j0": j0, "y0": y0, "yhat0": yh}
    if kind in ("self", "noalloc"):
        curve, (a, b) = _arc_curve(np.random.default_rng([11, int(seed) & 0x7FFFFFFF]))
        A = _self_matrix(_Arc(curve, 0, a, b), case["N"], case["kappa"])
        return A.T.contiguous()          # the library stores columns
    if kind == "served":
        ps = _requests(case, seed)
        if sum(_exact_cost(p) for p in ps) > 1.5e9:
            return None
        return [_exact_job(p)["traces"] for p in ps]
    p = _problem(case, seed)
    if _exact_cost(p) > 1.5e9:
        return None
    return _exact_job(p)


def _exact_cost(p):
    """Kernel evaluations, with the factorisations' loops, of the reference."""
    _, N = _sizes(p)
    nsum = N.astype(np.float64).sum(axis=0)
    return float((nsum * N[:, -1].sum()).sum() + 2e5 * N.size)


class _Arc:
    """x(t) = X(theta_c + half t) of a trigonometric curve, t in [-1, 1]."""

    def __init__(self, curve, ci, a, b):
        self.curve, self.ci, self.a, self.b = curve, ci, a, b
        self.c, self.half = 0.5 * (a + b), 0.5 * (b - a)
        self.next = self.prev = None

    def at_theta(self, th):
        th = np.asarray(th, dtype=np.float64)
        k = np.arange(len(self.curve["ax"]), dtype=np.float64)
        cs, sn = np.cos(th[..., None] * k), np.sin(th[..., None] * k)
        ax, bx, ay, by = (np.asarray(self.curve[n], dtype=np.float64) for n in ("ax", "bx", "ay", "by"))
        X = np.stack([cs @ ax + sn @ bx, cs @ ay + sn @ by], -1)
        D = np.stack([cs @ (k * bx) - sn @ (k * ax), cs @ (k * by) - sn @ (k * ay)], -1)
        return X, D

    def at(self, t):
        X, D = self.at_theta(self.c + self.half * np.asarray(t))
        return X, D * self.half

    def length(self):
        s, w = np.polynomial.legendre.leggauss(128)
        return float(w @ np.linalg.norm(self.at(s)[1], axis=-1))


def _wrap(a):
    r = np.mod(np.asarray(a) + math.pi, 2.0 * math.pi) - math.pi
    return np.where(r <= -math.pi, r + 2.0 * math.pi, r)


def _node_counts(o, length, om):
    if o["N_fixed"] > 0:
        return np.full(len(om), o["N_fixed"], dtype=np.int64)
    return np.maximum(o["N_min"], np.ceil(o["N_ppw"] * om * length - 1e-9).astype(np.int64) + o["N_off"])


def _cheb(n):
    return np.cos((2.0 * np.arange(n) + 1.0) * math.pi / (2.0 * n))


def _cutoff(x, lo, hi):
    """1 below lo, 0 above hi, exp(2 e^{-1/s} / (s - 1)) between."""
    x = np.abs(x)
    s = np.clip((x - lo) / (hi - lo), 1e-300, 1.0 - 1e-16)
    return np.where(x <= lo, 1.0, np.where(x >= hi, 0.0, np.exp(2.0 * np.exp(-1.0 / s) / (s - 1.0))))


def _chi(arc, t):
    """The partition of unity of a closed curve's overlapping arcs."""
    out = np.ones(t.shape)
    if arc.next is None:
        return out
    X, th = arc.at(t)[0], arc.c + arc.half * t
    for side in (1, -1):
        first, last = (arc, arc.next) if side > 0 else (arc.prev, arc)      # overlap [last.a, first.b]
        inside = (_wrap(th - last.a) >= 0.0) & (_wrap(first.b - th) >= 0.0) & (side * t > 0)
        end, far = arc.at_theta(first.b)[0], arc.at_theta(last.a)[0]
        A = float(np.linalg.norm(far - end))
        e = _cutoff(A - np.linalg.norm(X - end, axis=-1), A / 3.0, 2.0 * A / 3.0)
        out = np.where(inside, e if side > 0 else 1.0 - e, out)
    return out


def _dev(x):
    return torch.as_tensor(np.asarray(x), device="cuda" if torch.cuda.is_available() else "cpu")


def _bessel0(z):
    """J0 and Y0 in 64 bits (torch's own lose half the digits between 5 and 20): power series below 2, Miller's
    backward recurrence with Neumann's series for Y0 (DLMF 10.12.4, 10.8.2) up to 25, Hankel's expansion above."""
    zs, zm, zl = z.clamp(max=2.0), z.clamp(2.0, 25.0), z.clamp(min=25.0)
    u, term, harm = 0.25 * zs * zs, torch.ones_like(z), 0.0
    J, Yr = torch.ones_like(z), torch.zeros_like(z)
    for k in range(1, 19):
        term = term * (-u) / (k * k)
        harm += 1.0 / k
        J = J + term
        Yr = Yr - harm * term
    Y = (2.0 / math.pi) * ((torch.log(0.5 * zs) + np.euler_gamma) * J + Yr)
    hi, lo = torch.zeros_like(z), torch.full_like(z, 1e-100)      # J_{n+1}, J_n up to a factor
    norm, neumann = 2.0 * lo, lo / 30 * (-1) ** 30
    for n in range(60, 0, -1):
        hi, lo = lo, (2.0 * n / zm) * lo - hi
        if n % 2 == 1 and n > 1:
            norm = norm + 2.0 * lo
            neumann = neumann + lo * ((-1) ** ((n - 1) // 2) / ((n - 1) // 2))
    norm = norm + lo
    Jm = lo / norm
    Ym = (2.0 / math.pi) * (torch.log(0.5 * zm) + np.euler_gamma) * Jm - (4.0 / math.pi) * neumann / norm
    P, Qa, a = torch.ones_like(z), torch.zeros_like(z), torch.ones_like(z)
    for k in range(1, 20):
        a = a * ((2 * k - 1) ** 2 / (8.0 * k)) / zl
        if k % 2:
            Qa = Qa + a * (-1) ** ((k + 1) // 2)
        else:
            P = P + a * (-1) ** (k // 2)
    c, s, amp = torch.cos(zl), torch.sin(zl), torch.sqrt(1.0 / (math.pi * zl))
    cx, sx = c + s, s - c
    J = torch.where(z < 2.0, J, torch.where(z < 25.0, Jm, amp * (P * cx - Qa * sx)))
    Y = torch.where(z < 2.0, Y, torch.where(z < 25.0, Ym, amp * (P * sx + Qa * cx)))
    return J, Y


def _log_table(n):
    """int log|t_i - s| of the Lagrange basis over sqrt(1 - s^2), at the nodes themselves."""
    k = np.arange(1, n)
    T = _dev(np.cos(np.outer((2.0 * np.arange(n) + 1.0) * math.pi / (2.0 * n), k)))
    return -(math.pi / n) * (math.log(2.0) + 2.0 * (T / _dev(k.astype(np.float64))) @ T.T)


def _self_matrix(arc, n, kappa, table=None):
    t = _cheb(n)
    X, D = arc.at(t)
    Xd = _dev(X)
    R = torch.sqrt(((Xd[:, None] - Xd[None]) ** 2).sum(-1))
    dt = (_dev(t)[:, None] - _dev(t)[None]).abs()
    eye = torch.eye(n, dtype=torch.bool, device=R.device)
    z = torch.where(eye, torch.ones_like(R), kappa * R)
    J, Y = _bessel0(z)
    K1 = torch.where(eye, torch.full_like(J, -0.5 / math.pi), -J / (2.0 * math.pi))
    speed = _dev(np.log(0.5 * kappa * np.linalg.norm(D, axis=-1)))
    diag = -(np.euler_gamma + speed)[:, None].expand(n, n) / (2.0 * math.pi)
    re = torch.where(eye, diag, -0.25 * Y - K1 * torch.log(torch.where(eye, torch.ones_like(dt), dt)))
    im = torch.where(eye, torch.full_like(J, 0.25), 0.25 * J)
    w = math.pi / n
    return torch.complex(K1 * (_log_table(n) if table is None else table) + re * w, im * w)


def _near_weights(ts, n):
    """int log|t* - s| of the Lagrange basis over sqrt(1 - s^2) for |t*| > 1."""
    r = np.sqrt(ts * ts - 1.0)
    zeta = ts - np.sign(ts) * r
    k = np.arange(1, n)
    lam = np.concatenate([(math.pi * np.log(0.5 * (np.abs(ts) + r)))[:, None],
                          -(2.0 * math.pi / k) * zeta[:, None] ** k], axis=1)
    T = np.cos(np.outer(np.arange(n), (2.0 * np.arange(n) + 1.0) * math.pi / (2.0 * n)))
    return _dev(lam) @ _dev(T) / n


def _signal_at(sig, t):
    smp = sig.get("samples")
    if smp is None:
        return sig["amp"] * torch.sin(sig["carrier"] * t) * torch.exp(-(((t - sig["centre"]) / sig["width"]) ** 2))
    f, t0, dt = _dev(np.asarray(smp["f"], dtype=np.float64)), smp["t0"], smp["dt"]
    n = f.numel()
    s = (t - t0) / dt
    base = torch.floor(s)
    x = s - base + 3.0
    idx = base.long() - 3
    acc = torch.zeros_like(t)
    for k in range(8):
        w = torch.ones_like(x)
        for m in range(8):
            if m != k:
                w = w * (x - m) / (k - m)
        i = idx + k
        acc = acc + w * torch.where((i >= 0) & (i < n), f[i.clamp(0, n - 1)], torch.zeros_like(t))
    return torch.where((t >= t0) & (t <= t0 + (n - 1) * dt), acc, torch.zeros_like(t))


def _incident(sig, X, t):
    """u^i at points X and times t: a plane wave, or the retarded field of a point source by the trapezoid rule
    in v of f(t - r cosh v)."""
    t = _dev(t)
    if sig["kind"] == 1:
        return _signal_at(sig, t[None] - _dev(X @ np.asarray(sig["dir"]))[:, None])
    r = _dev(np.linalg.norm(X - np.asarray(sig["z0"]), axis=-1))[:, None]
    smp = sig.get("samples")
    first = smp["t0"] if smp else sig["centre"] - 8.0 * sig["width"]
    last = smp["t0"] + (len(smp["f"]) - 1) * smp["dt"] if smp else sig["centre"] + 8.0 * sig["width"]
    band = smp["band"] if smp else abs(sig["carrier"]) + 8.0 / sig["width"]
    out = torch.zeros(r.numel(), t.numel(), dtype=torch.float64, device=r.device)
    for c0 in range(0, t.numel(), 64):
        tc = t[None, c0:c0 + 64]
        hi, lo = (tc - first) / r, torch.clamp((tc - last) / r, min=1.0)
        on = hi > lo
        v0, v1 = torch.acosh(lo), torch.acosh(torch.where(on, hi, lo))
        n = int(((v1 - v0) * (1.25 * (band * r * torch.sinh(v1) + 1.0) + 24.0) / math.pi).max().item()) + 17
        acc = torch.zeros_like(v0)
        for k0 in range(0, n + 1, 256):
            k = torch.arange(k0, min(n + 1, k0 + 256), device=r.device, dtype=torch.float64)
            w = torch.where((k == 0) | (k == n), 0.5, 1.0)
            v = v0[..., None] + (v1 - v0)[..., None] * (k / n)
            acc += _signal_at(sig, tc[..., None] - r[..., None] * torch.cosh(v)) @ w.double()
        out[:, c0:c0 + 64] = torch.where(on, acc * (v1 - v0) / n / (2.0 * math.pi), torch.zeros_like(acc))
    return out


def _exact_job(p):
    """The discrete multiple-scattering iteration: densities summed over the steps, and the output traces."""
    o, sig = p["options"], p["signal"]
    L, Q, M, H, K = o["L"], o["Q"], o["M"], o["H"], o["n_period"]
    arcs = [_Arc(p["curves"][c], c, a, b) for c, a, b in p["arcs"]]
    P = len(arcs)
    for c in {a.ci for a in arcs}:
        ring = sorted((a for a in arcs if a.ci == c), key=lambda a: a.c % (2.0 * math.pi))
        for k, a in enumerate(ring if len(ring) > 1 else []):
            a.next, a.prev = ring[(k + 1) % len(ring)], ring[k - 1]
    h = o["W"] / (L - 1)
    om = np.arange(L) * h
    N = [_node_counts(o, a.length(), om) for a in arcs]
    nmax = [int(n[-1]) for n in N]
    # time grid, windows, phases e^{i omega_l (t_n - s_q)} with the integer part of the phase reduced exactly
    dt, s_q = 2.0 * math.pi / (h * K), 1.5 * H * np.arange(Q)
    NT = int((s_q[-1] + 2.0 * H) / dt) + 1
    t = -H + dt * np.arange(NT)
    u = t[None] - s_q[:, None]
    win = np.where(u >= -H / 2, _cutoff(u / H, 0.5, 1.0), 1.0 - _cutoff(u / H + 1.5, 0.5, 1.0))
    win = _dev(np.where(np.abs(u) >= H, 0.0, win))
    ln = _dev(np.mod(np.outer(np.arange(L), np.arange(NT)), K) * (2.0 * math.pi / K))
    fwd = [torch.polar(torch.ones_like(ln), _dev(np.arange(L) * (h * (-H - s)))[:, None] + ln) for s in s_q]
    wl_ = np.full(L, h)
    wl_[0], wl_[-1] = 0.0, 0.5 * h
    wl_ = _dev(wl_)
    valid = np.zeros((Q, NT), dtype=bool)
    for q in range(Q):
        n0 = int(math.ceil(s_q[q] / dt - 1e-9))
        valid[q, n0:n0 + K] = True
    valid = _dev(valid)

    def to_freq(g):                     # [n, NT] -> [n, Q, L]
        gc = g.to(torch.complex128)
        return torch.stack([dt * (gc * win[q]) @ fwd[q].T for q in range(Q)], 1)

    def to_time(V):                     # [n, Q, L] -> [n, NT]
        return sum(torch.where(valid[q], ((V[:, q] * wl_) @ fwd[q].conj()).real / math.pi,
                               torch.zeros((), dtype=torch.float64, device=V.device)) for q in range(Q))

    # targets: the transfer nodes of every arc, then the observation points
    tau = [_cheb(n) for n in nmax]
    chi = [_chi(a, x) for a, x in zip(arcs, tau)]
    obs = np.asarray(o["obs"], dtype=np.float64).reshape(-1, 2)
    tgt = np.concatenate([a.at(x)[0] for a, x in zip(arcs, tau)] + [obs])
    th = np.concatenate([a.c + a.half * x for a, x in zip(arcs, tau)] + [np.zeros(len(obs))])
    ci = np.concatenate([np.full(n, a.ci) for a, n in zip(arcs, nmax)] + [np.full(len(obs), -1)])
    off = np.concatenate([[0], np.cumsum(nmax)]).astype(int)
    live = np.concatenate([c > 0.0 for c in chi] + [np.ones(len(obs), dtype=bool)])
    param, keep, near = [], [], []
    for j, a in enumerate(arcs):
        ts = np.where(ci == a.ci, _wrap(th - a.c) / a.half, 9.0)
        on = live & ~((ci == a.ci) & (np.abs(ts) <= 1.0))
        on[off[j]:off[j + 1]] = False
        param.append(ts)
        keep.append(on)
        near.append(on & (ci == a.ci) & (np.abs(ts) <= 3.0))
    tgt_d = _dev(tgt)
    tables, weights, restr = {}, {}, {}

    def cross(l, j):                    # rows of arc j's potential at the kept targets
        n = int(N[j][l])
        x = _dev(arcs[j].at(_cheb(n))[0])
        R = torch.sqrt(((tgt_d[_dev(np.nonzero(keep[j])[0])][:, None] - x[None]) ** 2).sum(-1))
        z = om[l] * R
        J, Y = _bessel0(z)
        re, im = -0.25 * Y * (math.pi / n), 0.25 * J * (math.pi / n)
        nr = near[j][keep[j]]
        if nr.any():
            ts = param[j][keep[j]][nr]
            if (j, n) not in weights:
                weights[j, n] = (_near_weights(ts, n), torch.log((_dev(ts)[:, None] - _dev(_cheb(n))[None]).abs()))
            Wn, lg = weights[j, n]
            i = _dev(np.nonzero(nr)[0])
            K1 = -J[i] / (2.0 * math.pi)
            re[i] = K1 * Wn + (-0.25 * Y[i] - K1 * lg) * (math.pi / n)
        return torch.complex(re, im)

    E = {(l, j): cross(l, j) for l in range(1, L) for j in range(P)}
    lu = {}
    for j in range(P):
        for n in np.unique(N[j][1:]):
            tables.setdefault(int(n), _log_table(int(n)))
            ls = [l for l in range(1, L) if N[j][l] == n]
            for c0 in range(0, len(ls), 32):
                part = ls[c0:c0 + 32]
                A = torch.stack([_self_matrix(arcs[j], int(n), om[l], tables[int(n)]) for l in part])
                f, piv = torch.linalg.lu_factor(A)
                for i, l in enumerate(part):
                    lu[l, j] = (f[i], piv[i])

    def restrict(k, n):                 # transfer nodes -> n solve nodes
        if (n, nmax[k]) not in restr:
            kk = np.arange(1, nmax[k])
            a = np.cos(np.outer((2.0 * np.arange(n) + 1.0) * math.pi / (2.0 * n), kk))
            b = np.cos(np.outer((2.0 * np.arange(nmax[k]) + 1.0) * math.pi / (2.0 * nmax[k]), kk))
            restr[n, nmax[k]] = ((1.0 + 2.0 * _dev(a) @ _dev(b).T) / nmax[k]).to(torch.complex128)
        return restr[n, nmax[k]]

    data = [sig["sign"] * _dev(chi[k])[:, None] * _incident(sig, tgt[off[k]:off[k + 1]], t) for k in range(P)]
    total = {}
    Vobs = torch.zeros(len(obs), Q, L, dtype=torch.complex128, device=tgt_d.device)
    rows = [_dev(np.nonzero(k)[0]) for k in keep]
    for m in range(M):
        spec = [to_freq(g) for g in data]
        W = torch.zeros(len(tgt), Q, L, dtype=torch.complex128, device=tgt_d.device)
        for l in range(1, L):
            for j in range(P):
                phi = torch.linalg.lu_solve(*lu[l, j], restrict(j, int(N[j][l])) @ spec[j][:, :, l])
                total[l, j] = phi if m == 0 else total[l, j] + phi
                W[rows[j], :, l] += E[l, j] @ phi
        Vobs += W[off[P]:]
        if m + 1 < M:
            data = [-_dev(chi[k])[:, None] * to_time(W[off[k]:off[k + 1]]) for k in range(P)]
    tout = o["tout0"] + o["dtout"] * np.arange(o["n_tout"])
    tr = torch.zeros(len(obs), len(tout), dtype=torch.float64, device=tgt_d.device)
    for q in range(Q):
        rel = tout - s_q[q]
        ph = _dev(np.outer(np.arange(L), -h * rel))
        v = ((Vobs[:, q] * wl_) @ torch.polar(torch.ones_like(ph), ph)).real / math.pi
        tr += torch.where(_dev((rel >= -H) & (rel < 2.0 * math.pi / h - H)), v, torch.zeros_like(v))
    dens = [[torch.cat([total[l, j][:, q] for l in range(1, L)]).cpu() for q in range(Q)] for j in range(P)]
    if Q * P > 40:
        dens = [torch.cat(row) for row in dens]
    return {"traces": tr.cpu().numpy(), "densities": dens}
