"""The work that users of this library have it do, as measurable cases.

Every case goes through the public Python entry points (``Context``,
``Ensemble``, ``hermite_trajectory``, ``nb_force_few_noalloc``) on synthetic
Plummer spheres in N-body units, the input of the paper's experiments, with
the softenings and sizes of the benchmark's configurations.  A case is a dict
of plain values; ``prepare`` makes what a program has in hand before the call,
``run`` makes one pass, ``exact`` is the same result in plain 64-bit torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

import paper_cs_0702135_gb300 as nb
from paper_cs_0702135_gb300.autograd import hermite_trajectory

DEV = "cuda"
PAIR_FLOPS = 60          # the paper's count for one acc + jerk + pot interaction
VJP_FLOPS = 120          # its vector-Jacobian product: about twice that
STATE_BYTES = 108        # x, v, a, k (FP64), time and level of one particle
JREC_BYTES = 56          # m, x, v in FP64: what a force needs of one source
OUT_BYTES = 56           # acc, jerk, pot in FP64


def listed():
    return [
        # a small block of a block-step integration driven from the device:
        # latency counts (the median block at 2^16 bodies is of this order)
        {"name": "force_few", "kind": "force", "n": 65536, "na": 6, "inv_eps": 256, "host": False},
        # the mean block of the same run, through host arrays: a host integrator
        # that uses the library as the paper's host uses its GPU
        {"name": "force_block_host", "kind": "force", "n": 65536, "na": 1820, "inv_eps": 256, "host": True},
        # the full sweep of the headline benchmark
        {"name": "force_sweep", "kind": "force", "n": 1048576, "na": 1048576, "inv_eps": 1024, "host": False},
        # the all-FP64 force, the accuracy reference users run beside the fast one
        {"name": "force_fp64", "kind": "fp64", "n": 65536, "na": 1820, "inv_eps": 256},
        # reproducible GRAPE-style fixed-point sums, all particles active
        {"name": "force_fixed", "kind": "fixed", "n": 65536, "na": 65536, "inv_eps": 256},
        # the paper's comparison of summation orders, on a mean block
        {"name": "force_fp32", "kind": "fp32", "n": 65536, "na": 1820, "inv_eps": 256},
        {"name": "force_sorted", "kind": "sorted", "n": 65536, "na": 1820, "inv_eps": 256},
        # callers that may not allocate device memory; ragged size
        {"name": "force_noalloc", "kind": "noalloc", "n": 262181, "na": 64, "inv_eps": 256},
        # the paper's experiment at a small N: block steps from a checkpoint
        {"name": "run_1024", "kind": "run", "n": 1024, "inv_eps": 256, "level_min": 3},
        # ... and at its largest tabulated N of all machines, to a sixteenth
        {"name": "run_65536", "kind": "run", "n": 65536, "inv_eps": 256, "level_min": 4},
        # one step of fitting initial conditions through the integrator
        {"name": "trajectory_grad", "kind": "train", "n": 4096, "inv_eps": 256, "steps": 64, "ckpt": 8},
        # a stretch of an ensemble of clusters, with the energies and the state
        # a program writes out after it
        {"name": "ensemble", "kind": "ens", "clusters": 256, "n_lo": 32, "n_hi": 4096, "inv_eps": 256,
         "launches": 512},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["force", "force", "force", "fp64", "fixed", "fp32", "sorted", "noalloc", "run",
                       "run", "train", "ens"])
    c = {"kind": kind, "inv_eps": rng.choice([256, 1024])}
    if kind == "force":
        c["n"] = _log_int(rng, 256, 1 << 20)
        c["na"] = _log_int(rng, 1, c["n"])
        c["host"] = rng.random() < 0.5
    elif kind == "fp64":
        c["n"] = _log_int(rng, 256, 65536)
        c["na"] = _log_int(rng, 1, min(4096, c["n"]))
    elif kind == "fixed":
        c["n"] = _log_int(rng, 256, 131072)
        c["na"] = _log_int(rng, 1, c["n"])
    elif kind == "fp32":
        c["n"] = _log_int(rng, 256, 262144)
        c["na"] = _log_int(rng, 1, min(16384, c["n"]))
    elif kind == "sorted":
        c["n"] = _log_int(rng, 256, 262144)
        c["na"] = _log_int(rng, 1, min(2048, c["n"]))
    elif kind == "noalloc":
        c["n"] = _log_int(rng, 256, 1 << 20)
        c["na"] = rng.randint(1, 64)
    elif kind == "run":
        c["n"] = _log_int(rng, 128, 65536)
        c["level_min"] = rng.choice([3, 4])
        c["inv_eps"] = 256
    elif kind == "train":
        c["n"] = _log_int(rng, 128, 16384)
        c["steps"] = rng.randint(4, 64)
        c["ckpt"] = rng.randint(1, min(16, c["steps"]))
    else:
        c["clusters"] = _log_int(rng, 16, 512)
        c["n_lo"] = 32
        c["n_hi"] = _log_int(rng, 256, 4096)
        c["launches"] = rng.randint(64, 512)
        c["inv_eps"] = 256
    return c


# ----------------------------------------------------------------------------
# inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _direction(n, g):
    u = torch.rand((n, 2), generator=g, device=DEV, dtype=torch.float64)
    z = 1.0 - 2.0 * u[:, 0]
    rho = (1.0 - z * z).clamp_min(0.0).sqrt()
    phi = 2.0 * math.pi * u[:, 1]
    return torch.stack([rho * phi.cos(), rho * phi.sin(), z], dim=1)


def _plummer(n, g, m=None):
    """A Plummer sphere in N-body units, cut at 22.8 length units (on the GPU)."""
    q = torch.linspace(0.0, 1.0, 4097, device=DEV, dtype=torch.float64)
    pdf = q * q * (1.0 - q * q).clamp_min(0.0) ** 3.5
    cdf = torch.cumulative_trapezoid(pdf, q)
    cdf = torch.cat([torch.zeros(1, device=DEV, dtype=torch.float64), cdf / cdf[-1]])
    unit = 3.0 * math.pi / 16.0
    frac = (1.0 + (unit / 22.8) ** 2) ** -1.5          # enclosed mass inside the cut
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64).clamp_min(1e-12) * frac
    r = (u ** (-2.0 / 3.0) - 1.0) ** -0.5
    w = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    k = torch.searchsorted(cdf, w).clamp(1, 4096)
    t = (w - cdf[k - 1]) / (cdf[k] - cdf[k - 1]).clamp_min(1e-300)
    speed = (q[k - 1] + t * (q[k] - q[k - 1])) * math.sqrt(2.0) * (1.0 + r * r) ** -0.25
    x = _direction(n, g) * r[:, None] * unit
    v = _direction(n, g) * speed[:, None] / math.sqrt(unit)
    m = torch.full((n,), 1.0 / n, device=DEV, dtype=torch.float64) if m is None else m
    x = x - (m[:, None] * x).sum(0) / m.sum()
    v = v - (m[:, None] * v).sum(0) / m.sum()
    return m, x.contiguous(), v.contiguous()


def _system(case, seed):
    """(m, x, v) and the ascending active indices of a force case."""
    g = _gen(seed)
    n = case["n"]
    m, x, v = _plummer(n, g)
    na = case.get("na", n)
    idx = torch.randperm(n, generator=g, device=DEV)[:na].sort().values.to(torch.int32)
    return m, x, v, idx


def _clusters(case, seed):
    """Sizes log-uniform in [n_lo, n_hi] (the same for every seed), Salpeter masses; host arrays."""
    rs = np.random.RandomState(case["clusters"] * 4099 + case["n_hi"])
    lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"] + 1)
    sizes = np.clip(np.exp(rs.uniform(lo, hi, case["clusters"])).astype(np.int64), case["n_lo"], case["n_hi"])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    g = _gen(seed)
    big_m, big_x, big_v = _plummer(int(off[-1]), g)
    u = torch.rand(int(off[-1]), generator=g, device=DEV, dtype=torch.float64)
    s = (0.1 ** -1.35 + u * (100.0 ** -1.35 - 0.1 ** -1.35)) ** (-1.0 / 1.35)
    s, x, v = s.cpu().numpy(), big_x.cpu().numpy(), big_v.cpu().numpy()
    which = np.repeat(np.arange(len(sizes)), sizes)
    m = s / np.bincount(which, weights=s)[which]
    for c in range(3):
        x[:, c] -= np.bincount(which, weights=m * x[:, c])[which]
        v[:, c] -= np.bincount(which, weights=m * v[:, c])[which]
    return off, m, x, v


_SUM = {"fixed": nb.NB_SUM_FIXED, "fp32": nb.NB_SUM_FP32, "sorted": nb.NB_SUM_FP32_SORTED}


def prepare(case, seed):
    kind = case["kind"]
    eps = 1.0 / case["inv_eps"]
    st = {"case": case, "kind": kind, "eps": eps}
    if kind in ("force", "fp64", "fixed", "fp32", "sorted", "noalloc"):
        m, x, v, idx = _system(case, seed)
        torch.cuda.synchronize()
        na = case["na"]
        if kind == "noalloc":
            st.update(m=m, x=x, v=v)
        else:
            opts = {"flags": nb.NB_INIT_NO_FORCE, "summation": _SUM.get(kind, nb.NB_SUM_COMPENSATED),
                    "precision": nb.NB_FP64 if kind == "fp64" else nb.NB_DS}
            st["ctx"] = nb.Context.from_device(m, x, v, eps, **opts)
        if case.get("host"):
            st["idx"] = idx.cpu().numpy()
        else:
            st["idx"] = idx
            st["out"] = [torch.empty((na, 3), device=DEV, dtype=torch.float64),
                         torch.empty((na, 3), device=DEV, dtype=torch.float64),
                         torch.empty(na, device=DEV, dtype=torch.float64)]
    elif kind == "run":
        m, x, v, _ = _system(case, seed)
        torch.cuda.synchronize()
        st["ctx"] = nb.Context.from_device(m, x, v, eps, level_min=case["level_min"])
        st["start"] = st["ctx"].nb_get_state()
    elif kind == "train":
        m, x, v, _ = _system(case, seed)
        g = _gen(seed + 1)
        st["leaves"] = [t.requires_grad_(True) for t in (x, v, m)]
        st["grads"] = [torch.randn((case["n"], 3), generator=g, device=DEV, dtype=torch.float64) for _ in range(2)]
        torch.cuda.synchronize()
        st["stream"] = torch.cuda.Stream()
    else:
        off, m, x, v = _clusters(case, seed)
        st["ens"] = nb.Ensemble(off, m, x, v, eps)
        start = st["ens"].nb_ens_get_state()
        st["start"] = [start[k] for k in ("x", "v", "a", "k", "t", "level")]
    torch.cuda.synchronize()
    return st


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "noalloc":
        acc, jerk, pot = st["out"]
        nb.nb_force_few_noalloc(case["n"], st["m"], st["x"], st["v"], st["eps"], st["idx"], case["na"],
                                acc, jerk, pot, torch.cuda.current_stream().cuda_stream)
        return [acc, jerk, pot]
    if kind in ("force", "fp64", "fixed", "fp32", "sorted"):
        if case.get("host"):
            return list(st["ctx"].nb_force(st["idx"]))
        acc, jerk, pot = st["out"]
        st["ctx"].nb_force_dev(st["idx"], case["na"], acc, jerk, pot)
        return [acc, jerk, pot]
    if kind == "run":
        ctx, s = st["ctx"], st["start"]
        ctx.nb_set_state(s["x"], s["v"], s["a"], s["k"], s["t"], s["level"])
        steps, inter = ctx.nb_run(2.0 ** -case["level_min"])
        return {"state": ctx.nb_get_state(), "steps": steps, "interactions": inter}
    if kind == "train":
        x, v, m = st["leaves"]
        with torch.cuda.stream(st["stream"]):
            xt, vt = hermite_trajectory(x, v, m, st["eps"], 10, case["steps"], case["ckpt"])
            gx, gv, gm = torch.autograd.grad([xt, vt], [x, v, m], st["grads"])
        return [xt.detach(), vt.detach(), gx, gv, gm]
    ens = st["ens"]
    ens.nb_ens_set_state(*st["start"])
    launches, inter = ens.nb_ens_run(1.0, case["launches"])
    s = ens.nb_ens_get_state()
    ekin, epot = ens.nb_ens_energy()
    # the step and interaction counters of the state run on from pass to pass
    return {"state": [s[k] for k in ("x", "v", "a", "k", "t", "level")], "launches": launches,
            "interactions": inter, "ekin": ekin, "epot": epot}


# ----------------------------------------------------------------------------
# what a pass cannot do without

def _run_work(n, span):
    """Block steps of the paper's fits: n_steps = 247 N^0.35 a time unit, n_block = 0.20 N^0.81."""
    steps = 247.0 * n ** 0.35 * span
    block = min(float(n), 0.20 * n ** 0.81)
    return steps, block


def work(case):
    kind = case["kind"]
    if kind == "run":
        n = case["n"]
        steps, block = _run_work(n, 2.0 ** -case["level_min"])
        return {"bytes": 2 * STATE_BYTES * n, "flops": PAIR_FLOPS * steps * block * n}
    if kind == "train":
        n, steps = case["n"], case["steps"]
        return {"bytes": 2 * 7 * 8 * n + 96 * n * (steps // case["ckpt"] + 1),
                "flops": n * n * (PAIR_FLOPS * (2 * steps + 1) + VJP_FLOPS * (steps + 1))}
    if kind == "ens":
        # mean of n^2 for sizes log-uniform in [lo, hi]: the energies' pairs,
        # and one small block a launch for the steps
        lo, hi = case["n_lo"], case["n_hi"]
        n1 = (hi - lo) / math.log(hi / lo)
        n2 = 0.5 * (hi * hi - lo * lo) / math.log(hi / lo)
        c = case["clusters"]
        return {"bytes": 2 * STATE_BYTES * c * n1,
                "flops": c * (10 * n2 + PAIR_FLOPS * case["launches"] * 0.20 * n1 ** 0.81 * n1)}
    n, na = case["n"], case["na"]
    return {"bytes": JREC_BYTES * n + OUT_BYTES * na, "flops": PAIR_FLOPS * na * (n - 1)}


# ----------------------------------------------------------------------------
# the same in plain 64-bit torch

def _force64(m, x, v, eps, rows):
    """acc, jerk, pot on `rows` from all particles; the self pair is left out."""
    out = []
    n = m.shape[0]
    chunk = max(1, (1 << 25) // n)
    for s in range(0, rows.shape[0], chunk):
        i = rows[s:s + chunk]
        d = [x[None, :, c] - x[i, None, c] for c in range(3)]
        w = [v[None, :, c] - v[i, None, c] for c in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps
        own = torch.zeros_like(r2, dtype=torch.bool).scatter_(1, i[:, None], True)
        rinv = torch.where(own, torch.zeros_like(r2), r2.rsqrt())
        mr = m[None, :] * rinv
        mr3 = mr * rinv * rinv
        b = -3.0 * (d[0] * w[0] + d[1] * w[1] + d[2] * w[2]) * rinv * rinv
        out.append((torch.stack([(mr3 * d[c]).sum(1) for c in range(3)], 1),
                    torch.stack([(mr3 * (w[c] + b * d[c])).sum(1) for c in range(3)], 1), -mr.sum(1)))
    return [torch.cat([o[k] for o in out]) for k in range(3)]


def _trajectory64(x, v, m, eps, dt, steps):
    rows = torch.arange(m.shape[0], device=x.device)

    def force(x, v, m):
        return tuple(_force64(m, x, v, eps, rows)[:2])

    ck = torch.utils.checkpoint.checkpoint
    a, k = ck(force, x, v, m, use_reentrant=False)
    for _ in range(steps):
        xp = x + (v + (dt / 2) * (a + (dt / 3) * k)) * dt
        vp = v + (a + (dt / 2) * k) * dt
        an, kn = ck(force, xp, vp, m, use_reentrant=False)
        a3 = 2.0 * (a - an) + (k + kn) * dt
        a2 = -3.0 * (a - an) - (2.0 * k + kn) * dt
        x, v, a, k = xp + (a2 / 12 + a3 / 20) * dt * dt, vp + (a2 / 3 + a3 / 4) * dt, an, kn
    return x, v


def exact(case, seed):
    kind, eps = case["kind"], 1.0 / case["inv_eps"]
    if kind in ("run", "ens"):
        # block steps of individual particles: a trajectory whose step levels
        # follow the sums' last bits has no single 64-bit value
        return None
    m, x, v, idx = _system(case, seed)
    if kind == "train":
        n = case["n"]
        if n > 8192 or n * n * case["steps"] > 4e9:
            return None
        g = _gen(seed + 1)
        gx, gv = [torch.randn((n, 3), generator=g, device=DEV, dtype=torch.float64) for _ in range(2)]
        leaves = [t.requires_grad_(True) for t in (x, v, m)]
        xt, vt = _trajectory64(x, v, m, eps, 2.0 ** -10, case["steps"])
        return [xt.detach(), vt.detach(), *torch.autograd.grad([xt, vt], leaves, [gx, gv])]
    if case["n"] * case["na"] > 2e10:
        return None
    return _force64(m, x, v, eps, idx.long())
