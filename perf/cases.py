"""Workloads that time the framework through its public entry points.

Each case is one of the jobs the library is used for, with inputs of the laws that
`paper_2607_24741_b200/workloads.py` describes, drawn here on the GPU from a seed:

  solve     create -> drain -> potentials, depths, residuals -> close, on device tensors
  host      sinkhorn_batch_solve_host: the whole call on pinned host buffers
  refill    a queue of problems through fewer slots, new ones replacing finished ones
  apply     the plan of a finished batch applied to point values (barycentric images)
  residual  the row residual of potentials that the caller already holds

Outputs are the potentials, the completion depth and status of every lane and its achieved
two-sided residual.  The column residual alone is not among them: after a g-leg the column
marginal is exact up to rounding (Eq. 4), so its value is rounding noise.
"""
from __future__ import annotations

import ctypes
import math

import torch

from paper_2607_24741_b200 import binding as B

DEV = "cuda:0"

# Cycles that a typical lane of the law needs at its tolerance (used for the operation counts only).
TYPICAL_CYCLES = {"tiny": 340, "sensor": 6, "feature": 370, "registration": 280, "sweep": 580}


def listed():
    return [
        # a handful of small two-dimensional problems: nothing but latency and launches
        dict(name="tiny", job="solve", law="tiny", W=8, n=64, m=64, d=2, tol=1e-3, max_iter=5000, mode="active"),
        # a day of sensor windows, one coupling per window (z-scored features, uneven weights)
        dict(name="sensor", job="solve", law="sensor", W=256, n=512, m=512, d=15, tol=1e-3, max_iter=5000, mode="active"),
        # the same from a program whose data lives on the host, a few windows of uneven length
        dict(name="sensor_host", job="host", law="sensor", W=16, n=200, m=264, d=15, tol=1e-3, max_iter=5000, mode="active"),
        # minibatch couplings of bf16 embeddings inside a training loop, with an iteration budget
        dict(name="feature", job="solve", law="feature", W=64, n=1024, m=1024, d=512, tol=1e-3, max_iter=100, mode="active"),
        # smaller embeddings, ragged minibatches
        dict(name="feature_d128", job="solve", law="feature", W=24, n=500, m=333, d=128, tol=1e-3, max_iter=100, mode="active"),
        # point-cloud registration, the largest job one GPU is given
        dict(name="registration", job="solve", law="registration", W=32, n=8192, m=8192, d=3, tol=1e-3, max_iter=5000, mode="active"),
        # one pair of scans by itself
        dict(name="registration_one", job="solve", law="registration", W=1, n=4096, m=4096, d=3, tol=1e-3, max_iter=5000, mode="active"),
        # lanes whose regularisations, and so completion depths, differ widely
        dict(name="sweep", job="solve", law="sweep", W=1024, n=256, m=256, d=8, tol=1e-3, max_iter=50000, mode="active"),
        # the logical-mask control on such lanes, ragged
        dict(name="sweep_masked", job="solve", law="sweep", W=96, n=100, m=77, d=8, tol=3e-3, max_iter=5000, mode="masked"),
        # a queue of such problems through a quarter of the slots
        dict(name="sweep_refill", job="refill", law="sweep", W=256, n=128, m=160, d=8, tol=3e-3, max_iter=5000, mode="active"),
        # images of the points under the plan of a finished registration
        dict(name="apply", job="apply", law="registration", W=8, n=4096, m=4096, d=3, tol=1e-2, max_iter=5000, mode="active"),
        # audit of potentials that another program stored
        dict(name="residual", job="residual", law="sensor", W=32, n=1024, m=1000, d=15, tol=1e-3, max_iter=5000, mode="active"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    law = rng.choice(["tiny", "sensor", "feature", "registration", "sweep", "sweep"])
    job, mode, tol, max_iter = "solve", "active", 1e-3, 5000
    if law == "tiny":
        W, n, m, d = _log(rng, 2, 64), _log(rng, 16, 128), _log(rng, 16, 128), 2
    elif law == "sensor":
        job = rng.choice(["solve", "solve", "host", "residual"])
        W, n, m, d = _log(rng, 4, 256), _log(rng, 100, 512), _log(rng, 100, 512), rng.randint(9, 16)
        if job == "residual":
            W, n, m = _log(rng, 4, 64), _log(rng, 100, 1024), _log(rng, 100, 1024)
    elif law == "feature":
        W, n, m = _log(rng, 2, 64), _log(rng, 128, 1024), _log(rng, 128, 1024)
        d, max_iter = rng.choice([64, 128, 256, 320, 512]), rng.choice([20, 50, 100])
    elif law == "registration":
        job = rng.choice(["solve", "solve", "solve", "apply"])
        n = _log(rng, 500, 8192)
        W, m, d = max(1, min(_log(rng, 1, 32), (16 * 8192 * 8192) // (n * n))), n, 3
        if job == "apply":
            W, tol = min(W, 8), 1e-2
    else:
        job = rng.choice(["solve", "solve", "refill"])
        mode = "active" if job == "refill" else rng.choice(["active", "active", "masked", "static"])
        W, n, m, d = _log(rng, 16, 512), _log(rng, 32, 256), _log(rng, 32, 256), rng.randint(4, 8)
        tol = rng.choice([1e-2, 3e-3]) if job == "refill" or mode != "active" else rng.choice([1e-2, 3e-3, 1e-3])
    return dict(job=job, law=law, W=W, n=n, m=m, d=d, tol=tol, max_iter=max_iter, mode=mode)


# ------------------------------------------------------------------------------- inputs

def _inputs(case, seed):
    """x [W,n,d], y [W,m,d], a [W,n], b [W,m], eps [W] on the GPU, rounded once to the storage type."""
    W, n, m, d, law = case["W"], case["n"], case["m"], case["d"], case["law"]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1000003 * int(seed) + 17)
    normal = lambda *s: torch.randn(*s, generator=gen, device=DEV, dtype=torch.float32)
    uniform = lambda *s: torch.rand(*s, generator=gen, device=DEV, dtype=torch.float32)
    a, b = torch.full((W, n), 1.0 / n, device=DEV), torch.full((W, m), 1.0 / m, device=DEV)
    if law == "tiny":
        mu, s = 2.0 * uniform(W, 1, d), 0.5 + 1.5 * uniform(W, 1, 1)
        x, y = normal(W, n, d), mu + s.sqrt() * normal(W, m, d)
        eps = torch.full((W,), 0.05, device=DEV)
    elif law == "sensor":
        delta, u = 0.3 * normal(W, 1, d), uniform(W, 1, d)
        x, y = normal(W, n, d), delta + (1.0 + 0.5 * u).sqrt() * normal(W, m, d)
        # Dirichlet(5): a gamma variable of shape 5 is a sum of five exponentials
        a = -torch.log(1.0 - uniform(5, W, n)).double().sum(0)
        b = -torch.log(1.0 - uniform(5, W, m)).double().sum(0)
        a, b = (a / a.sum(1, keepdim=True)).float(), (b / b.sum(1, keepdim=True)).float()
        eps = 0.1 * torch.cdist(x, y).square().flatten(1).median(dim=1).values
    elif law == "feature":
        mu = normal(W, 10, d)
        pick = lambda k: torch.gather(mu, 1, torch.randint(10, (W, k, 1), generator=gen, device=DEV).expand(W, k, d))
        unit = lambda v: v / v.norm(dim=2, keepdim=True)
        x = unit(normal(W, n, d) + pick(n)).bfloat16()
        y = unit(normal(W, m, d) + pick(m)).bfloat16()
        eps = torch.full((W,), 0.05, device=DEV)
    elif law == "registration":
        v = normal(W, n, d)
        x = v / v.norm(dim=2, keepdim=True) * (1.0 + 0.02 * normal(W, n, 1))
        q, r = torch.linalg.qr(normal(W, d, d).double())
        q = q * torch.sign(torch.diagonal(r, dim1=1, dim2=2))[:, None, :]
        q[:, :, 0] *= torch.sign(torch.linalg.det(q))[:, None]
        y = x @ q.transpose(1, 2).float() + 0.01 * normal(W, n, d)
        y = torch.where(uniform(W, n, 1) < 0.10, 2.0 * uniform(W, n, d) - 1.0, y)
        a, b = 0.5 + uniform(W, n).double(), 0.5 + uniform(W, n).double()
        a, b = (a / a.sum(1, keepdim=True)).float(), (b / b.sum(1, keepdim=True)).float()
        eps = torch.full((W,), 0.01, device=DEV)
    else:
        x, y = normal(W, n, d), normal(W, m, d)
        eps = torch.exp(math.log(0.01) + (math.log(0.5) - math.log(0.01)) * uniform(W))
    return x.contiguous(), y.contiguous(), a, b, eps.contiguous()


def _solve(case, p, **kw):
    return B.SinkhornBatch(*p, case["tol"], mode=case["mode"], max_iter=case["max_iter"], **kw)


def _results(sb):
    f, g = sb.potentials()
    depth, status = sb.depths()
    r_row, r_col = sb.residuals()
    # lanes that the iteration limit stopped before a column check have no r_col (NaN)
    return {"f": f, "g": g, "depth": depth, "status": status, "residual": torch.fmax(r_row, r_col)}


def prepare(case, seed):
    p = _inputs(case, seed)
    st = {"case": case, "inputs": p}
    W, n, m, d = case["W"], case["n"], case["m"], case["d"]
    if case["job"] == "host":
        st["host"] = [t.cpu().pin_memory() for t in p]
        cfg = B.make_config(W, n, m, d, mode=case["mode"], max_iter=case["max_iter"],
                            stream=torch.cuda.current_stream().cuda_stream)
        need = B.sinkhorn_batch_host_workspace_bytes(cfg)
        st["workspace"] = torch.empty(need, dtype=torch.uint8, device=DEV)
        cfg.workspace, cfg.workspace_bytes = st["workspace"].data_ptr(), need
        st["cfg"] = cfg
        pinned = lambda *s, dt=torch.float32: torch.zeros(*s, dtype=dt).pin_memory()
        st["out"] = {"f": pinned(W, n), "g": pinned(W, m), "depth": pinned(W, dt=torch.int32),
                     "status": pinned(W, dt=torch.int32), "r_row": pinned(W), "r_col": pinned(W)}
    elif case["job"] == "apply":
        st["batch"] = _solve(case, p)                    # the finished batch that the program keeps
        st["batch"].drain()
        st["values"] = p[1].float()
    elif case["job"] == "residual":
        sb = _solve(case, p)
        sb.drain()
        st["potentials"] = sb.potentials(f64=True)
        sb.close()
    return st


def run(state):
    case, p = state["case"], state["inputs"]
    job = case["job"]
    if job == "solve":
        sb = _solve(case, p)
        sb.drain()
        out = _results(sb)
        sb.close()
        return out
    if job == "host":
        x, y, a, b, eps = (t.data_ptr() for t in state["host"])
        o = state["out"]
        slots, cycles = ctypes.c_longlong(0), ctypes.c_int(0)
        rc = B.lib.sinkhorn_batch_solve_host(x, y, a, b, eps, case["tol"], ctypes.byref(state["cfg"]),
                                             o["f"].data_ptr(), o["g"].data_ptr(), o["depth"].data_ptr(),
                                             o["status"].data_ptr(), o["r_row"].data_ptr(), o["r_col"].data_ptr(),
                                             ctypes.byref(slots), ctypes.byref(cycles))
        if rc != B.SKB_OK:
            raise B.SkbError(rc, B.lib.sinkhorn_batch_last_error(None).decode())
        return {"f": o["f"], "g": o["g"], "depth": o["depth"], "status": o["status"],
                "residual": torch.fmax(o["r_row"], o["r_col"])}
    if job == "refill":
        W = case["W"]
        slots = max(1, W // 4)
        sb = _solve(case, [t[:slots] for t in p], lane_capacity=W)
        taken = slots
        while taken < W:
            sb.step(16)
            free = min(slots - sb.active(), W - taken)
            if free * 8 >= slots or free == W - taken > 0:
                sb.refill(*(t[taken:taken + free] for t in p))
                taken += free
        sb.drain()
        out = _results(sb)
        sb.close()
        return out
    if job == "apply":
        return state["batch"].apply_plan(state["values"])
    x, y, a, b, eps = p
    f, g = state["potentials"]
    return B.sinkhorn_row_residual_static(x, y, a, f, g, eps)


def work(case):
    """One pass cannot do without: the costs once (2 d operations per pair), two multiply-adds per pair
    and cycle (one in each leg), the inputs read and the results written once."""
    W, n, m, d = case["W"], case["n"], case["m"], case["d"]
    pairs = W * n * m
    el = 2 if case["law"] == "feature" else 4
    moved = W * (n + m) * d * el + W * (n + m) * 4 + 4 * W
    if case["job"] == "apply":
        return {"bytes": moved + W * (n + m) * 8 + 4 * W * (n + m) * d, "flops": pairs * (2 * d + 4 + 2 * d)}
    if case["job"] == "residual":
        return {"bytes": moved + W * (n + m) * 8 + 4 * W, "flops": pairs * (2 * d + 4)}
    cycles = min(case["max_iter"], TYPICAL_CYCLES[case["law"]])
    return {"bytes": moved + W * (n + m) * 4 + 12 * W, "flops": pairs * (2 * d + 4 * cycles)}


def tolerance(case):
    if case["job"] == "apply":
        return {"rel": 1e-6, "max": 1e-4}              # float64 sums, stored as fp32
    if case["job"] == "residual":
        return {"rel": 1e-6}
    # Depths: a lane may stop one audit later or earlier when its residual passes the tolerance
    # within the arithmetic's rounding; every lane that does moves its potentials by one cycle.
    # Measured against 64 bits: potentials 2e-8 .. 4e-6, residuals 2e-6 .. 1.1e-4 (fp32 exponents).
    if case["law"] == "feature":
        return {"rel": 1e-4, "max": 1e-2, "differ": 0.01}
    return {"rel": 5e-4, "max": 1e-2, "differ": 0.01}


# ------------------------------------------------------------------------------- 64-bit values

def _solve64(x, y, a, b, eps, tol, max_iter, static):
    """Alternating updates of Eq. 3 in float64 for a few lanes at a time: log domain for the first cycles,
    then scalings against a plan that is formed anew every few cycles (so that nothing leaves the range)."""
    x, y, a, b, eps = (t.double() for t in (x, y, a, b, eps))
    sq = lambda t: t.square().sum(2)
    S = (sq(x)[:, :, None] + sq(y)[:, None, :] - 2.0 * torch.bmm(x, y.transpose(1, 2))) / eps[:, None, None]
    W, n, m = S.shape
    phi, gam = torch.zeros(W, n, 1, device=DEV, dtype=torch.float64), torch.zeros(W, 1, m, device=DEV, dtype=torch.float64)
    u, v = torch.ones_like(phi), torch.ones_like(gam).transpose(1, 2)
    la, lb = torch.log(a)[:, :, None], torch.log(b)[:, None, :]
    f, g = torch.zeros_like(a), torch.zeros_like(b)
    depth = torch.zeros(W, dtype=torch.int32, device=DEV)
    status, resid = torch.zeros_like(depth), torch.full((W,), float("nan"), device=DEV, dtype=torch.float64)
    P, k = None, 0

    def keep(now, st, k):
        f[now] = (eps[:, None] * (phi + torch.log(u))[:, :, 0])[now]
        g[now] = (eps[:, None] * (gam[:, 0, :] + torch.log(v)[:, :, 0]))[now]
        if st:
            depth[now], status[now] = k, st

    warm = 12
    while True:
        if k < warm:
            fresh = la - torch.logsumexp(gam - S, dim=2, keepdim=True)
            marginal = a * torch.exp(phi - fresh)[:, :, 0]
        else:
            rows = torch.bmm(P, v)
            marginal = (u * rows)[:, :, 0]
        if k:
            r = (marginal - a).abs().sum(1)
            resid = torch.where(status == 0, r, resid)
            keep((status == 0) & (r <= tol), 1, k)
            last = k == max_iter
            if last:
                keep(status == 0, 2, k)
            if (last or k % 8 == 0 or W == 1 or static) and bool((status != 0).all()):
                if static:                                # every lane is carried on to the deepest lane's cycle
                    every = torch.ones(W, dtype=torch.bool, device=DEV)
                    keep(every, 0, k)
                    resid = r
                break
        if k < warm:
            phi = fresh
            gam = lb - torch.logsumexp(phi - S, dim=1, keepdim=True)
        else:
            u = a[:, :, None] / rows
            v = b[:, :, None] / torch.bmm(P.transpose(1, 2), u)
        k += 1
        if k >= warm and (k - warm) % 12 == 0:
            phi, gam = phi + torch.log(u), gam + torch.log(v).transpose(1, 2)
            u, v = torch.ones_like(u), torch.ones_like(v)
            P = torch.exp(phi + gam - S)
    return f, g, depth, status, resid


def exact(case, seed):
    p = _inputs(case, seed)
    W, n, m = case["W"], case["n"], case["m"]
    if case["job"] in ("apply", "residual"):
        st = prepare(case, seed)
        x, y, a, b, eps = p
        f, g = st["batch"].potentials(f64=True) if case["job"] == "apply" else st["potentials"]
        out = []
        for t in range(W):
            P = torch.exp((f[t][:, None] + g[t][None, :] - torch.cdist(
                x[t].double(), y[t].double(), compute_mode="donot_use_mm_for_euclid_dist").square()) / eps[t].double())
            out.append(P @ y[t].double() if case["job"] == "apply" else (P.sum(1) - a[t].double()).abs().sum())
        return torch.stack(out)
    static = case["mode"] == "static"
    step = W if static else max(1, (1 << 27) // (n * m))
    parts = [_solve64(*(t[i:i + step] for t in p), case["tol"], case["max_iter"], static) for i in range(0, W, step)]
    f, g, depth, status, resid = (torch.cat(c) for c in zip(*parts))
    return {"f": f, "g": g, "depth": depth, "status": status, "residual": resid}
