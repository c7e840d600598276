"""The calls a user of this library makes, as measurable cases.

Every case is one pass of the library's ordinary flow on a context that holds a batch: draw the
initial condition (``reset``), integrate every trajectory to its last step, reduce (``results``)
and, where the case says so, read the trajectories back (``state``) or run the adjoint
(``backward``).  Shapes are those of ``workloads.py`` and ``bench.py``, with step counts cut so
that a pass stays short where only the length of the run would differ.

A case is {"kind", "sets", "traj", "steps", ...}: ``sets`` parameter sets of ``traj``
trajectories and ``steps`` steps each (``ragged`` > 0: sizes and step counts spread
log-uniformly down to 1/``ragged`` of those, drawn from ``sizes``).  Parameters and noise come
from the seed given to ``prepare``.
"""
import math
import random

import numpy as np
import torch

from paper_1104_2499_gb300 import abp, workloads

DT = 1e-3
_stream = None


def _case(name, kind, sets, traj, steps, **kw):
    c = dict(kind=kind, sets=sets, traj=traj, steps=steps, ragged=1, sizes=0, bins=0, snap=0, K=0, window=0, heun=False,
             xorshift=False, fp64=False, v0=0, state=False)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the paper's work items, one trajectory per parameter value: the smallest call, all latency
        _case("items_64", "items", 64, 1, 1_000),
        # as many one-trajectory work items as fill the chip once
        _case("items_8192", "items", 8_192, 1, 1_000),
        # the largest of the time-against-work-items curve
        _case("items_65536", "items", 65_536, 1, 4_000),
        # one parameter set with its position histogram, the first thing anyone runs
        _case("single_4096", "single", 1, 4_096, 10_000, bins=256),
        # the flagship: the D x q grid, 2,097,152 trajectories
        _case("sweep_2048x1024", "grid", 2_048, 1_024, 20_000, bins=256, v0=1),
        # sets of uneven size and length, none a multiple of a block
        _case("uneven_512", "uneven", 512, 16_384, 100_000, ragged=64, sizes=2, bins=256),
        # mean velocity against the load (the paper's Fig. 2)
        _case("load_64x4096", "load", 64, 4_096, 10_000),
        # the second-order scheme over a grid
        _case("heun_512x1024", "grid", 512, 1_024, 10_000, heun=True, v0=1),
        # the paper's own generator over a grid
        _case("xorshift_512x1024", "grid", 512, 1_024, 10_000, xorshift=True, v0=1),
        # a large ensemble watched while it runs: position and velocity histograms
        _case("snapshots_4M", "single", 1, 4_194_304, 4_000, bins=1_024, snap=500),
        # forward and windowed pathwise adjoint (over longer windows the derivative itself explodes):
        # one optimisation step on the parameters
        _case("gradient_262144", "gradient", 1, 262_144, 4_000, K=1_000, window=1_000),
        # the FP64 state, run when single precision is to be checked
        _case("fp64_4096", "single", 1, 4_096, 1_000, fp64=True, state=True, v0=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["items", "single", "grid", "grid", "uneven", "load", "gradient", "snapshots", "fp64"])
    if kind == "items":
        return _case("", "items", _log(rng, 1, 65_536), 1, _log(rng, 250, 4_000))
    if kind == "single":
        steps = _log(rng, 500, 10_000)
        return _case("", "single", 1, _log(rng, 1, 65_536), steps, bins=rng.choice([0, 256]), heun=rng.random() < 0.25,
                     state=steps <= 4_000, v0=rng.randint(0, 1))
    if kind == "grid":
        mode = rng.choice(["em", "em", "heun", "xorshift"])
        return _case("", "grid", _log(rng, 16, 2_048), _log(rng, 64, 1_024), _log(rng, 1_000, 10_000),
                     bins=rng.choice([0, 256]), heun=mode == "heun", xorshift=mode == "xorshift", v0=1)
    if kind == "uneven":
        return _case("", "uneven", _log(rng, 8, 512), _log(rng, 1_000, 16_384), _log(rng, 5_000, 100_000), ragged=64,
                     sizes=rng.randrange(1 << 20), bins=rng.choice([0, 256]))
    if kind == "load":
        return _case("", "load", _log(rng, 8, 64), _log(rng, 256, 4_096), _log(rng, 1_000, 10_000))
    if kind == "gradient":
        K = rng.choice([64, 200, 333, 500, 1_000])
        steps = _log(rng, 500, 4_000)
        return _case("", "gradient", _log(rng, 1, 64), _log(rng, 256, 4_096), steps, ragged=rng.choice([1, 4]),
                     sizes=rng.randrange(1 << 20), K=K, window=0 if steps <= 1_000 else K * (1_000 // K), v0=rng.randint(0, 1))
    if kind == "snapshots":
        steps = _log(rng, 500, 4_000)
        return _case("", "single", 1, _log(rng, 65_536, 4_194_304), steps, bins=rng.choice([64, 1_000, 1_024]),
                     snap=max(1, steps // rng.randint(2, 8)))
    return _case("", "single", 1, _log(rng, 256, 4_096), _log(rng, 250, 1_000), fp64=True, state=True, v0=rng.randint(0, 1))


def _sizes(case):
    """Trajectories and steps of every set (they do not depend on the seed)."""
    n = case["sets"]
    if case["ragged"] <= 1:
        return [case["traj"]] * n, [case["steps"]] * n
    r = np.random.default_rng(case["sizes"])
    f = np.exp(-r.uniform(0.0, math.log(case["ragged"]), (2, n)))
    return ([max(1, int(v)) for v in np.rint(case["traj"] * f[0])], [max(1, int(v)) for v in np.rint(case["steps"] * f[1])])


def _params(case, seed):
    """The parameter sets: the ranges of workloads.py, placed by the seed."""
    n, r = case["sets"], np.random.default_rng(seed)
    base = [dict(workloads.DEFAULTS) for _ in range(n)]
    if case["kind"] == "items":
        for p, D in zip(base, np.exp(r.uniform(math.log(1e-2), 0.0, n))):
            p["D"] = float(D)
    elif case["kind"] == "single":
        base[0]["D"] = float(r.uniform(0.1, 0.2))
    elif case["kind"] == "grid":
        D, q = np.exp(r.uniform(math.log(1e-3), 0.0, n)), np.exp(r.uniform(math.log(0.1), math.log(10.0), n))
        for i, p in enumerate(base):
            p["D"], p["q"] = float(D[i]), float(q[i])
    elif case["kind"] == "uneven":
        D, a = np.exp(r.uniform(math.log(1e-3), 0.0, n)), r.uniform(0.0, 0.5, n)
        for i, p in enumerate(base):
            p["D"], p["asym"] = float(D[i]), float(a[i])
    elif case["kind"] == "load":
        for p, F in zip(base, np.linspace(-1.0, 1.0, n) + r.uniform(-0.01, 0.01)):
            p["F0"] = float(F)
    else:
        for p, D in zip(base, r.uniform(0.05, 0.2, n)):
            p["D"] = float(D)
    return base


def _workload(case, seed):
    M, N = _sizes(case)
    return workloads.Workload(name=case["kind"], sets=_params(case, seed), n_traj=M, n_steps=N, dt=DT, seed=seed, v0_mode=case["v0"],
                              hist_x_bins=case["bins"], hist_v_bins=case["bins"] if case["snap"] else 0,
                              snapshot_every=case["snap"], checkpoint_every=case["K"], scheme=1 if case["heun"] else 0,
                              noise=1 if case["xorshift"] else 0)


def prepare(case, seed):
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    ens = abp.Ensemble(_workload(case, seed), stream=_stream, state_fp64=case["fp64"])
    ens.set_params()
    return {"ens": ens, "case": case}


def run(state):
    ens, case = state["ens"], state["case"]
    with torch.cuda.stream(_stream):
        ens.reset()
        ens.integrate()
        out = ens.results()
        if case["state"]:
            out.update(ens.state())
        if case["K"]:
            out["grad"] = ens.backward(window=case["window"])
    return out


def work(case):
    """Parameters in, results out; operations: 35 FP32 lane operations per particle-step of the
    Euler-Maruyama step and its noise, 51 of the Heun step, and for the adjoint one more forward
    step and a reverse step of 44."""
    M, N = _sizes(case)
    steps = sum(m * n for m, n in zip(M, N))
    per = 51 if case["heun"] else 35
    if case["K"]:
        per += 35 + 44
    n_snap = max(N) // case["snap"] if case["snap"] else 1
    nbytes = case["sets"] * (72 + 64) + n_snap * case["sets"] * 4 * case["bins"] * (2 if case["snap"] else 1)
    if case["state"]:
        nbytes += 40 * sum(M)
    if case["K"]:
        nbytes += 48 * case["sets"]
    return {"bytes": nbytes, "flops": per * steps}


# ------------------------------------------------------------------ the same in 64 bits

_M32 = 0xFFFFFFFF


def _philox(c, k0, k1):
    """Philox4x32-10 on int64 tensors of 32-bit words."""
    c0, c1, c2, c3 = c
    for _ in range(10):
        # 32 x 32 -> 64-bit products in two halves, so that nothing leaves int64's range
        h0, l0 = _mul(0xD2511F53, c0)
        h1, l1 = _mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _mul(a, b):
    lo = a * (b & 0xFFFF)
    hi = a * (b >> 16) + (lo >> 16)
    return (hi >> 16) & _M32, ((hi << 16) | (lo & 0xFFFF)) & _M32


def _normals(wa, wb):
    r = torch.sqrt(-2.0 * torch.log((wa.double() + 0.5) * 2.0 ** -32))
    a = (wb >> 9).double() * (2.0 ** -23 * 2.0 * math.pi)
    return r * torch.cos(a), r * torch.sin(a)


def _xorshift(s):
    t = s[0] ^ ((s[0] << 11) & _M32)
    w = s[3] ^ (s[3] >> 19) ^ t ^ (t >> 8)
    return [s[1], s[2], s[3], w], w


def exact(case, seed):
    M, N = _sizes(case)
    T, n_max = sum(M), max(N)
    # about 0.4 ms a step for the launches of plain torch, and the arithmetic of large ensembles
    if n_max * (8e-4 + 8e-10 * T) * (3 if case["K"] else 1) > 15.0:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    f64 = dict(dtype=torch.float64, device=dev)
    P = _params(case, seed)
    set_of = torch.repeat_interleave(torch.arange(len(M), device=dev), torch.tensor(M, device=dev))
    p = {k: torch.tensor([s[k] for s in P], **f64)[set_of] for k in workloads.PARAM_NAMES}
    n_of = torch.tensor(N, device=dev)[set_of]
    t = torch.arange(T, device=dev, dtype=torch.int64)
    zero, k0, k1 = torch.zeros_like(t), seed & _M32, (seed >> 32) & _M32
    w = _philox((zero, zero + 0x80000000, t, zero), k0, k1)
    x0 = p["L"] * ((w[0] >> 8).double() * 2.0 ** -24)
    z0 = _normals(w[1], w[2])[0]
    x, v = x0.clone(), torch.sqrt(p["D"]) * z0 if case["v0"] else torch.zeros(T, **f64)
    e = torch.zeros(T, **f64)
    if case["xorshift"]:
        xs = list(_philox((zero + 1, zero + 0x80000000, t, zero), k0, k1))
    B = p["h"] * 0.453 * 2.0 * math.pi / p["L"]
    sig = torch.sqrt(2.0 * p["D"] * DT)

    def drift(x, v, e):
        ph = 2.0 * math.pi * (x / p["L"] + 0.1903)
        dv = (p["d"] * e - p["gamma0"]) * v + p["F0"] + B * (torch.cos(ph) + 2.0 * p["asym"] * torch.cos(2.0 * ph))
        return ph, dv * DT, (p["q"] - p["c"] * e - p["d"] * e * v * v) * DT

    grad = None
    if case["K"]:
        # tangents of (x, v, e) with respect to (D, q, c, d, gamma0, asym), the noise held fixed
        tx, tv, te, acc = (torch.zeros((6, T), **f64) for _ in range(4))
        if case["v0"]:
            tv[0] = z0 / (2.0 * torch.sqrt(p["D"]))
    ragged, z = min(N) < n_max, None
    for n in range(n_max):
        if case["xorshift"]:
            xs, wa = _xorshift(xs)
            xs, wb = _xorshift(xs)
            zn = _normals(wa, wb)[0]
        else:
            if n % 4 == 0:
                w = _philox((zero + (n >> 2), zero, t, zero), k0, k1)
                z = _normals(w[0], w[1]) + _normals(w[2], w[3])
            zn = z[n % 4]
        s = sig * zn
        ph, dv, de = drift(x, v, e)
        if case["heun"]:
            vp, ep = v + dv + s, e + de
            _, dv1, de1 = drift(x + v * DT, vp, ep)
            nx, nv, ne = x + 0.5 * (v + vp) * DT, v + 0.5 * (dv + dv1) + s, e + 0.5 * (de + de1)
        else:
            nx, nv, ne = x + v * DT, v + dv + s, e + de
        if case["K"]:
            if case["window"] and n % case["window"] == 0 and n:
                tx, tv, te = torch.zeros_like(tx), torch.zeros_like(tv), torch.zeros_like(te)
            fx = -B * (2.0 * math.pi / p["L"]) * (torch.sin(ph) + 4.0 * p["asym"] * torch.sin(2.0 * ph)) * DT
            ntv = tv * (1.0 + DT * (p["d"] * e - p["gamma0"])) + tx * fx + te * (DT * p["d"] * v)
            nte = te * (1.0 - DT * p["c"] - DT * p["d"] * v * v) - tv * (2.0 * DT * p["d"] * e * v)
            ntx = tx + tv * DT
            ntv[0] += s / (2.0 * p["D"])
            nte[1] += DT
            nte[2] -= DT * e
            ntv[3] += DT * e * v
            nte[3] -= DT * e * v * v
            ntv[4] -= DT * v
            ntv[5] += DT * B * 2.0 * torch.cos(2.0 * ph)
            acc = torch.where(n < n_of, acc + tv, acc) if ragged else acc + tv
        if ragged:
            on = n < n_of
            nx, nv, ne = torch.where(on, nx, x), torch.where(on, nv, v), torch.where(on, ne, e)
            if case["K"]:
                ntx, ntv, nte = torch.where(on, ntx, tx), torch.where(on, ntv, tv), torch.where(on, nte, te)
        x, v, e = nx, nv, ne
        if case["K"]:
            tx, tv, te = ntx, ntv, nte
    Td = n_of.double() * DT
    dx = x - x0
    vbar = dx / Td

    def per_set(a):
        return torch.zeros(len(M), **f64).index_add_(0, set_of, a)

    Md, Tset = torch.tensor(M, **f64), torch.tensor(N, **f64) * DT
    sums = [per_set(a) for a in (vbar, vbar * vbar, dx, dx * dx)]
    mean = sums[0] / Md
    dev2 = per_set((vbar - mean[set_of]) ** 2)
    se = torch.where(Md > 1, torch.sqrt(dev2 / torch.clamp(Md - 1.0, min=1.0) / Md), torch.zeros_like(Md))
    msd = sums[3] / Md
    out = {"moments": torch.stack([mean, se, msd, (msd - (sums[2] / Md) ** 2) / (2.0 * Tset)] + sums, 1)}
    if case["bins"]:
        out["hist_x"] = None
        if case["snap"]:
            out["hist_v"] = None
    if case["state"]:
        out.update(x=x, x0=x0, v=v, e=e, vbar=vbar)
    if case["K"]:
        grad = torch.stack([per_set(acc[j] / n_of.double()) / Md for j in range(6)], 1)
        out["grad"] = grad
    return out
