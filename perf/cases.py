"""Cases of the solver's performance measurement, through its public Python API.

Each listed case is one call (or one batch of calls) that a user makes: a full
solve (pruning, domain selection, reconstruction), a domain-selection session,
a batch of energies, or a batch of requests to the server. Sizes, restart
counts and coupling families are those of the benchmark's workloads, the tests
and the serving stream; long runs take fewer steps than a production solve,
with the same work per step. `draw` gives further cases over the same ranges.

listed() / draw(rng)   cases: dicts of plain values
prepare(case, seed)    a user's inputs (made from the seed) and handles
run(state)             one pass; returns its whole outputs
exact(case, seed)      the same outputs in FP64 where they have such a value
work(case)             bytes and operations one pass cannot do without
"""

from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2312_05837_gb300 import api

# Restart-steps whose state (theta, m, v: 12 bytes each) cannot stay on the
# chip (registers, shared and tensor memory of all SMs, about 100 MB) are read
# and written once per step.
ON_CHIP_BYTES = 100e6

_ctx = None


def _context() -> api.Context:
    """One library context for the process, as a program keeps it."""
    global _ctx
    if _ctx is None:
        _ctx = api.Context(0)
    return _ctx


def listed() -> list[dict]:
    return [
        # the smallest call: a 100-spin glass from host memory (latency, launches)
        dict(name="sk100", op="solve", family="sk", n=100, dtype="f64", mem="host",
             restarts=64, steps=1000),
        # max-cut on a mid-size random graph, dense +-1 couplings (exact 8-bit operands)
        dict(name="er2000", op="solve", family="er_dense", n=2000, degree=10.0, dtype="i8",
             mem="device", restarts=1024, steps=2000),
        # complete graph with uniform couplings and fields (two operand planes)
        dict(name="complete1000", op="solve", family="complete", n=1000, dtype="f32",
             mem="device", restarts=1024, steps=1000),
        # the largest dense solve: a 4096-spin glass with fields, 4096 restarts
        dict(name="sk4096", op="solve", family="sk_h", n=4096, dtype="f32", mem="device",
             restarts=4096, steps=1000),
        # the same kind in the faster, row-scaled 8-bit precision, odd sizes
        dict(name="sk3001_fp8", op="solve", family="sk_h", n=3001, dtype="f32", mem="device",
             restarts=2000, steps=500, precision="fp8"),
        # sparse +-1 lattice
        dict(name="torus20k", op="solve", family="torus", n=20000, dtype="i8", mem="device",
             restarts=512, steps=1000),
        # the largest sparse solve: random graph with pendant trees that pruning removes
        dict(name="er120k_trees", op="solve", family="er_trees", n=120000, degree=4.0, dtype="i8",
             mem="device", restarts=512, steps=300),
        # a sparse request of the serving stream, alone
        dict(name="er997", op="solve", family="er", n=997, degree=8.0, dtype="i8", mem="device",
             restarts=256, steps=2000),
        # early retirement: 6-regular graph, real couplings, the convergence rule
        dict(name="regular1000_conv", op="session", family="regular", n=1000, degree=6.0,
             dtype="f64", mem="device", restarts=1024, steps=1000, converge=True),
        # the plain FP32 form (reference precision) as a session
        dict(name="sk1500_fp32", op="session", family="sk_h", n=1500, dtype="f32", mem="device",
             restarts=512, steps=100, precision="fp32"),
        # energies of many spin vectors
        dict(name="energy4096", op="energy", family="sk_h", n=4096, dtype="f32", mem="device",
             count=256),
        # a batch of requests to the server: half dense glasses, half sparse graphs
        dict(name="serve24", op="serve", n=4096, n_min=64, requests=24, restarts=256, steps=1000),
    ]


def _log(rng, lo, hi) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    """One more case of the ranges above (odd sizes included)."""
    op = rng.choice(["dense", "dense", "dense", "sparse", "sparse", "sparse", "session", "energy",
                     "serve"])
    if op == "dense":
        family = rng.choice(["sk", "sk_h", "er_dense", "complete"])
        n, B = _log(rng, 40, 4096), _log(rng, 16, 4096)
        steps = max(50, min(2000, int(2e13 / (n * n * B)), int(2e9 / (n * B))))
        c = dict(op="solve", family=family, n=n, mem=rng.choice(["device", "device", "host"]),
                 dtype="i8" if family == "er_dense" else rng.choice(["f32", "f64"]),
                 restarts=B, steps=steps)
        if family == "er_dense":
            c["degree"] = rng.uniform(4.0, 12.0)
        elif rng.random() < 0.3:
            c["precision"] = "fp8"
        return c
    if op == "sparse":
        family = rng.choice(["er", "er", "torus", "er_trees", "regular"])
        n, B = _log(rng, 64, 120000), _log(rng, 16, 512)
        if family == "torus":
            side = max(4, int(math.sqrt(n)))
            n = side * max(4, n // side)
        n += n % 2 if family == "regular" else 0
        steps = max(50, min(2000, int(4e9 / (n * B))))
        return dict(op="solve", family=family, n=n, degree=rng.uniform(3.0, 9.0),
                    dtype="f64" if family == "regular" else "i8", mem=rng.choice(["device", "host"]),
                    restarts=B, steps=steps)
    if op == "session":
        n, B = _log(rng, 100, 2000), _log(rng, 16, 1024)
        if rng.random() < 0.5:
            return dict(op="session", family="regular", n=n + n % 2, degree=6.0, dtype="f64",
                        mem="device", restarts=B, steps=1000, converge=True)
        return dict(op="session", family="sk_h", n=n, dtype="f32", mem="device", restarts=B,
                    steps=max(20, min(200, int(1e11 / (n * n * B)))), precision="fp32")
    if op == "energy":
        family = rng.choice(["sk_h", "er_dense", "er", "complete"])
        n = _log(rng, 64, 20000 if family == "er" else 5000)
        return dict(op="energy", family=family, n=n, degree=8.0, mem="device",
                    dtype="i8" if family in ("er_dense", "er") else rng.choice(["f32", "f64"]),
                    count=_log(rng, 1, 512))
    return dict(op="serve", n=_log(rng, 500, 4096), n_min=64, requests=rng.randrange(4, 25),
                restarts=rng.choice([128, 200, 256]), steps=rng.randrange(200, 1001))


# ------------------------------------------------------------------ instances

_NP = {"f64": torch.float64, "f32": torch.float32, "i8": torch.int8}


def _csr(n, lo, hi, w):
    """Symmetric CSR (int64 offsets, int32 columns, values) of distinct edges lo < hi."""
    rows, cols, vals = torch.cat([lo, hi]), torch.cat([hi, lo]), torch.cat([w, w])
    order = torch.argsort(rows * n + cols)
    rows, cols, vals = rows[order], cols[order], vals[order]
    indptr = torch.zeros(n + 1, dtype=torch.int64, device=rows.device)
    indptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return indptr, cols.to(torch.int32).contiguous(), vals.contiguous()


def _distinct(n, a, b):
    """Distinct pairs lo < hi of a list of vertex pairs (loops dropped)."""
    keep = a != b
    key = torch.unique(torch.minimum(a, b)[keep] * n + torch.maximum(a, b)[keep])
    return key // n, key % n


def _random_edges(n, degree, g, base=None):
    """About n * degree / 2 distinct edges of a uniform random graph on the first `base` vertices."""
    base = base or n
    m = int(base * min(degree, base - 1) / 2)
    a = torch.randint(0, base, (m,), generator=g, device="cuda")
    b = torch.randint(0, base, (m,), generator=g, device="cuda")
    return _distinct(n, a, b)


def _pm1(m, g):
    return (2 * torch.randint(0, 2, (m,), generator=g, device="cuda") - 1).to(torch.int8)


def _instance(case, seed, family=None, n=None):
    """A seeded instance of the case's family, on the device."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    family, n = family or case["family"], n or case["n"]
    dt = _NP[case.get("dtype", "f32")]
    kw = dict(n=n, J=None, indptr=None, indices=None, data=None, h=None, j_scale=1.0,
              convention="physics")
    if family in ("sk", "sk_h", "complete"):
        if family == "complete":  # couplings and fields U(-1000, 1000), the paper's convention
            x = torch.rand(n, n, generator=g, device="cuda", dtype=dt) * 2000.0 - 1000.0
            kw.update(h=torch.rand(n, generator=g, device="cuda", dtype=dt) * 2000.0 - 1000.0,
                      j_scale=0.5, convention="paper")
        else:
            x = torch.randn(n, n, generator=g, device="cuda", dtype=dt) / math.sqrt(n)
            if family == "sk_h":
                kw["h"] = torch.randn(n, generator=g, device="cuda", dtype=dt) * math.sqrt(0.1)
        J = torch.triu(x, 1)
        return SimpleNamespace(**{**kw, "layout": "dense", "J": (J + J.T).contiguous()})
    if family == "er_dense":  # max-cut: J = -W, W = +-1 on the edges, cut weight 1/2
        lo, hi = _random_edges(n, case["degree"], g)
        w = _pm1(lo.numel(), g)
        J = torch.zeros(n, n, dtype=torch.int8, device="cuda")
        J[lo, hi] = w
        J[hi, lo] = w
        return SimpleNamespace(**{**kw, "layout": "dense", "J": J, "j_scale": 0.5})
    if family == "torus":
        rows = max(4, int(math.sqrt(n / 2)) if n == 20000 else int(math.sqrt(n)))
        idx = torch.arange(n, device="cuda").reshape(rows, n // rows)
        a = torch.cat([idx.reshape(-1), idx.reshape(-1)])
        b = torch.cat([idx.roll(-1, 1).reshape(-1), idx.roll(-1, 0).reshape(-1)])
        lo, hi = _distinct(n, a, b)
    elif family == "er_trees":  # a sixth of the spins in trees of depth <= 3 on the others
        base = n - n // 6
        lo, hi = _random_edges(n, case["degree"], g, base)
        extra = torch.arange(base, n, device="cuda")
        d1, d2 = base + (n - base + 1) // 2, base + (n - base + 1) * 5 // 6
        u = torch.rand(n - base, generator=g, device="cuda", dtype=torch.float64)
        first = torch.where(extra < d1, 0, torch.where(extra < d2, base, d1))
        count = torch.where(extra < d1, base, torch.where(extra < d2, d1 - base, max(1, d2 - d1)))
        parent = torch.minimum(first + (u * count).long(), extra - 1)
        lo, hi = _distinct(n, torch.cat([lo, parent]), torch.cat([hi, extra]))
    elif family == "regular":  # union of three random Hamiltonian cycles: degree 6 but for repeats
        ps = [torch.randperm(n, generator=g, device="cuda") for _ in range(3)]
        lo, hi = _distinct(n, torch.cat(ps), torch.cat([p.roll(-1) for p in ps]))
    else:
        lo, hi = _random_edges(n, case["degree"], g)
    if family == "regular":  # couplings and fields U(-1, 1)
        w = torch.rand(lo.numel(), generator=g, device="cuda", dtype=dt) * 2.0 - 1.0
        kw.update(h=torch.rand(n, generator=g, device="cuda", dtype=dt) * 2.0 - 1.0, j_scale=0.5,
                  convention="paper")
    else:
        w = _pm1(lo.numel(), g)
    kw["indptr"], kw["indices"], kw["data"] = _csr(n, lo, hi, w)
    return SimpleNamespace(**{**kw, "layout": "csr"})


def _to_host(inst):
    return SimpleNamespace(**{k: v.cpu().numpy() if isinstance(v, torch.Tensor) else v
                              for k, v in vars(inst).items()})


def _spins(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
    bits = torch.randint(0, 2, (case["count"], case["n"]), generator=g, device="cuda")
    return (2 * bits - 1).to(torch.int8)


def _requests(case, seed):
    """(instance, precision) of each request: sizes log-spaced in [n_min, n],
    dense and sparse in turn."""
    k = case["requests"]
    out = []
    for r in range(k):
        n = int(round(case["n_min"] * (case["n"] / case["n_min"]) ** (r / max(1, k - 1))))
        dense = r % 2 == 0
        inst = _instance(dict(dtype="f32", degree=8.0), seed * 1009 + r,
                         "sk_h" if dense else "er", n)
        out.append((_to_host(inst), "fp8" if dense else "auto"))
    return out


# ------------------------------------------------------------------ the calls

def prepare(case, seed):
    ctx = _context()
    st = dict(case=case, ctx=ctx, seed=int(seed) & 0xFFFF)
    if case["op"] == "serve":
        st["requests"] = _requests(case, seed)
        st["server"] = api.Server(ctx, budget_bytes=64 << 30, max_active=32, chunk_steps=100,
                                  pack=True)
        return st
    inst = _instance(case, seed)
    st["inst"] = _to_host(inst) if case["mem"] == "host" else inst
    if case["op"] == "energy":
        st["spins"] = _spins(case, seed)
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    if case["op"] == "energy":
        return api.energy(ctx, st["inst"], st["spins"])
    kw = dict(seed=st["seed"], precision=case.get("precision", "auto"),
              converge=case.get("converge", False))
    if case["op"] == "solve":
        r = api.solve(ctx, st["inst"], case["restarts"], case["steps"], **kw)
        return {k: r[k] for k in ("best_spins", "best_energy", "best_restart", "best_step")}
    if case["op"] == "session":
        s = api.Session(ctx, st["inst"], case["restarts"], case["steps"], **kw)
        s.run(case["steps"])
        s.finish()
        E, step, spins = s.restart_best(device=True)
        out = dict(energies=E, steps=step, spins=spins)
        if case.get("converge"):
            out["stopped"] = s.convergence()
        s.close()
        return out
    srv = st["server"]
    kw.pop("precision"), kw.pop("converge")
    ids = [srv.submit(inst, case["restarts"], case["steps"], precision=prec, **kw)
           for inst, prec in st["requests"]]
    got = [srv.wait(i) for i in ids]
    for i in ids:
        srv.release(i)
    return dict(energies=np.array([g["best_energy"] for g in got]),
                spins=np.concatenate([g["best_spins"] for g in got]),
                restarts=np.array([g["best_restart"] for g in got]),
                steps=np.array([g["best_step"] for g in got]))


def exact(case, seed):
    """Energies in FP64; the search's own outputs (which restart wins, at which
    step, with which spins) follow a chaotic trajectory and have no such value."""
    if case["op"] != "energy":
        return None
    inst, s = _instance(case, seed), _spins(case, seed).double()
    cq, ch = (inst.j_scale, 1.0) if inst.convention == "paper" else (-0.5 * inst.j_scale, -1.0)
    if inst.layout == "dense":
        E = cq * ((s @ inst.J.double()) * s).sum(1)
    else:
        rows = torch.repeat_interleave(torch.arange(inst.n, device="cuda"), inst.indptr.diff())
        E = torch.stack([cq * (inst.data.double() * v[rows] * v[inst.indices.long()]).sum() for v in s])
    return E + ch * (s @ inst.h.double()) if inst.h is not None else E


def _shape(case, n=None, family=None):
    """(stored couplings, bytes of one with its column) of an instance."""
    n, family = n or case["n"], family or case["family"]
    size = {"f64": 8, "f32": 4, "i8": 1}[case.get("dtype", "f32")]
    if family in ("sk", "sk_h", "complete", "er_dense"):
        return float(n) * n, size
    degree = {"torus": 4.0, "regular": 6.0}.get(family, case.get("degree", 8.0))
    return n * min(degree, n - 1), size + 4


def work(case):
    """Each coupling and spin vector once, two operations per coupling and
    restart-step (about 30 more per spin for the update); the state of a step
    only where it cannot stay on the chip."""
    if case["op"] == "energy":
        nnz, size = _shape(case)
        return dict(bytes=nnz * size + case["count"] * (case["n"] + 8.0),
                    flops=2.0 * nnz * case["count"])
    B, T = case["restarts"], case["steps"]
    if case.get("converge"):
        T = min(T, 64)  # a restart stops after about this many steps on average
    if case["op"] == "serve":
        k, nb, fl = case["requests"], 0.0, 0.0
        for r in range(k):
            n = int(round(case["n_min"] * (case["n"] / case["n_min"]) ** (r / max(1, k - 1))))
            nnz, size = _shape(dict(dtype="f32" if r % 2 == 0 else "i8", degree=8.0), n,
                               "sk_h" if r % 2 == 0 else "er")
            nb += nnz * size + n
            fl += (2.0 * nnz + 30.0 * n) * B * T
        return dict(bytes=nb, flops=fl)
    n = case["n"]
    nnz, size = _shape(case)
    state = 24.0 * n * B * T if 12.0 * n * B > ON_CHIP_BYTES else 0.0
    return dict(bytes=nnz * size + n + state, flops=(2.0 * nnz + 30.0 * n) * B * T)
