"""Performance cases: what a user of this package has it compute, through its public calls.

Every case is one call (or the two or three calls that belong together) of
paper_2406_05061_gb300.native on clouds shaped like the ones the package's workloads
draw. Sinkhorn loops run a fixed number of iterations (tau = 0), so that a pass does the
same work whatever the rounding; entropic maps take potentials made here. ``exact``
restates each case in float64 with plain torch.
"""
import math
import random

import numpy as np
import torch

from paper_2406_05061_gb300 import native, workloads

# eps schedules run from BETA0 eps0 down to S_LAST eps0, eps0 = mean cost / 20, along the
# constant-speed progress t_k (the shape of the package's automatic schedule)
BETA0, S_LAST = 5.0, 0.3


def listed():
    return [
        # the smallest solve: the 2-D Gaussian pair on which everything else is checked, default precision
        dict(name="sinkhorn_2d_512", kind="sinkhorn", cloud="gauss2", n=512, m=512, d=2, iters=40, weights=False,
             precision="fp32"),
        # out-of-sample points mapped with stored potentials (a query against a fitted map), default precision
        dict(name="map_query_1000", kind="map", cloud="gmm", n=1000, m=2048, d=16, K=4, precision="fp32"),
        # cell-response experiments: about 11k against 2.8k cells, 47 features, default precision
        dict(name="progot_11000x2800_d47", kind="progot", cloud="gmm", n=11000, m=2800, d=47, K=4, iters=8,
             weights=False, precision="fp32"),
        # a coupling and its report (transport cost, entropy, both marginals), default precision
        dict(name="coupling_8192_d64", kind="coupling", cloud="gmm", n=8192, m=8192, d=64, iters=10,
             precision="fp32"),
        # the benchmark's Sinkhorn solve, mixed precision
        dict(name="sinkhorn_8192_d64_mixed", kind="sinkhorn", cloud="gmm", n=8192, m=8192, d=64, iters=100,
             weights=False, precision="bf16x3"),
        # a small served request: uneven clouds with weights, mixed precision
        dict(name="progot_1777x3001_d16_mixed", kind="progot", cloud="gmm", n=1777, m=3001, d=16, K=4, iters=20,
             weights=True, precision="bf16x3"),
        # embeddings on the sphere: the wide, large solve, mixed precision
        dict(name="sinkhorn_20000x16384_d256_mixed", kind="sinkhorn", cloud="sphere", n=20000, m=16384, d=256,
             iters=8, weights=False, precision="bf16x3"),
        # a whole data set carried through a fitted K-step map, mixed precision
        dict(name="map_10007_d64_mixed", kind="map", cloud="gmm", n=10007, m=8192, d=64, K=8, precision="bf16x3"),
        # the same for embeddings
        dict(name="map_16384x32768_d256_mixed", kind="map", cloud="sphere", n=16384, m=32768, d=256, K=2,
             precision="bf16x3"),
        # grey images against their blurs (32 x 32 pixels), mixed precision
        dict(name="progot_images_6000_mixed", kind="progot", cloud="images", n=6000, m=6000, d=1024, K=2, iters=5,
             weights=False, precision="bf16x3"),
        # many uneven problems solved together
        dict(name="batch_64_mixed", kind="batch", count=64, lo=128, hi=4096, sizes=3, K=4, iters=20,
             precision="bf16x3"),
        # the p-norm ground cost of the coupling experiments
        dict(name="progot_pnorm_11000x2800", kind="pnorm", cloud="gmm", n=11000, m=2800, d=47, p=1.5, K=2, iters=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["sinkhorn", "sinkhorn", "map", "map", "progot", "progot", "coupling", "images", "batch", "pnorm"])
    precision = rng.choice(["fp32", "bf16x3"])
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(8, 64), lo=128, hi=_log_int(rng, 512, 4096),
                    sizes=rng.randint(0, 10**6), K=rng.choice([2, 4]), iters=rng.randint(4, 20), precision="bf16x3")
    if kind == "pnorm":
        return dict(kind="pnorm", cloud="gmm", n=_log_int(rng, 300, 11000), m=_log_int(rng, 300, 2800),
                    d=_log_int(rng, 3, 47), p=rng.choice([1.5, 1.5, 1.25, 3.0]), K=rng.choice([1, 2]),
                    iters=rng.randint(2, 5))
    if kind == "images":
        n = _log_int(rng, 500, 6000)
        return dict(kind="progot", cloud="images", n=n, m=n, d=rng.choice([400, 576, 784, 1024]), K=rng.choice([1, 2]),
                    iters=rng.randint(2, 5), weights=False, precision="bf16x3")
    d = _log_int(rng, 2, 256)
    n, m = _log_int(rng, 300, 20000), _log_int(rng, 300, 20000)
    cloud = "sphere" if d > 64 else "gmm"
    if kind == "map":
        return dict(kind="map", cloud=cloud, n=n, m=m, d=d, K=rng.randint(1, 8 if d <= 64 else 2), precision=precision)
    if kind == "coupling":
        return dict(kind="coupling", cloud=cloud, n=min(n, 10000), m=min(m, 10000), d=d, iters=rng.randint(4, 12),
                    precision=precision)
    if kind == "sinkhorn":
        iters = rng.randint(10, 100) if max(n, m) * d < 400000 else rng.randint(4, 8)
        return dict(kind="sinkhorn", cloud=cloud, n=n, m=m, d=d, iters=iters, weights=rng.random() < 0.3,
                    precision=precision)
    K = rng.choice([2, 4])
    iters = rng.randint(4, 20) if max(n, m) * d < 400000 else rng.randint(1, 3)
    return dict(kind="progot", cloud=cloud, n=n, m=m, d=d, K=K, iters=iters, weights=rng.random() < 0.3,
                precision=precision)


# ---------------------------------------------------------------- inputs
def _clouds(case, seed):
    n, m, d, cloud = case["n"], case["m"], case["d"], case["cloud"]
    if cloud == "gauss2":
        pr = workloads.gaussian_affine(n, m, seed=seed)
    elif cloud == "sphere":
        pr = workloads.sphere_mixture_pair(n, m, d, seed=seed)
    elif cloud == "images":
        pr = workloads.blur_pair(n, math.isqrt(d), 2.0, seed=seed)
    else:
        pr = workloads.gmm_pair(n, m, d, seed=seed)
    return pr.x, pr.y


def _mean_cost(x, y):
    x, y = x.astype(np.float64), y.astype(np.float64)
    c = (x * x).sum(1).mean() + (y * y).sum(1).mean() - 2.0 * float(x.mean(0) @ y.mean(0))
    return float("%.6g" % c)


def _mean_cost_p(x, y, p):
    """Mean p-norm cost over a sample of pairs (only a scale for eps)."""
    k = min(len(x), len(y), 2048)
    return float("%.6g" % (np.abs(x[:k].astype(np.float64) - y[:k]) ** p).sum(1).mean()) / p


def _alpha(K):
    return [1.0 / (K - k) for k in range(K)]


def _eps(K, eps0):
    return [(1.0 - (k + 1) / K) * BETA0 * eps0 + (k + 1) / K * S_LAST * eps0 for k in range(K)]


def _weights(rng, n):
    w = rng.uniform(0.5, 1.5, n)
    return (w / w.sum()).astype(np.float32)


def _host_inputs(case, seed):
    """Clouds, weights and schedules of a single-problem case (numpy)."""
    x, y = _clouds(case, seed)
    rng = np.random.default_rng(seed + 77)
    h = dict(x=x, y=y, a=None, b=None)
    if case.get("weights"):
        h["a"], h["b"] = _weights(rng, case["n"]), _weights(rng, case["m"])
    K = case.get("K", 1)
    eps0 = (_mean_cost_p(x, y, case["p"]) if case["kind"] == "pnorm" else _mean_cost(x, y)) / 20.0
    h["eps"] = _eps(K, eps0) if "K" in case else [0.5 * eps0]
    h["alpha"] = _alpha(K)
    return h


def _batch_sizes(case):
    """Log-uniform n and m, d of 16 or 64 (the shapes are the case's, the points the seed's)."""
    rng = random.Random(case["sizes"])
    return [(_log_int(rng, case["lo"], case["hi"]), _log_int(rng, case["lo"], case["hi"]), rng.choice([16, 64]))
            for _ in range(case["count"])]


def _batch_inputs(case, seed):
    out = []
    for i, (n, m, d) in enumerate(_batch_sizes(case)):
        pr = workloads.gmm_pair(n, m, d, seed=1000 * seed + i)
        out.append(dict(x=pr.x, y=pr.y, eps=_eps(case["K"], _mean_cost(pr.x, pr.y) / 20.0), alpha=_alpha(case["K"]),
                        a=None, b=None))
    return out


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _stored_potentials(h, dev):
    """g of every step as a fit would have left it: a few float64 updates against a sample of x."""
    y = torch.from_numpy(h["y"]).to(dev).double()
    x = torch.from_numpy(h["x"][:1024]).to(dev).double()
    rows = []
    for eps in h["eps"]:
        C = _sq_cost(x, y)
        g = torch.zeros(len(y), dtype=torch.float64, device=dev)
        for _ in range(4):
            f = -eps * torch.logsumexp((g[None, :] - C) / eps, 1) - eps * math.log(len(x))
            g = -eps * torch.logsumexp((f[:, None] - C) / eps, 0) - eps * math.log(len(y))
        rows.append(g.float())
    return torch.stack(rows)


# ---------------------------------------------------------------- the pass
def prepare(case, seed):
    dev = _device()
    kind = case["kind"]
    if kind == "batch":
        probs = [dict(p, x=torch.from_numpy(p["x"]).to(dev), y=torch.from_numpy(p["y"]).to(dev),
                      tau=[0.0] * case["K"]) for p in _batch_inputs(case, seed)]
        return dict(case=case, plan=native.BatchPlan(probs, max_iter=case["iters"], precision=case["precision"]))
    h = _host_inputs(case, seed)
    s = dict(case=case, alpha=np.array(h["alpha"]), eps=np.array(h["eps"]), tau=np.zeros(len(h["eps"])))
    for k in ("x", "y", "a", "b"):
        s[k] = None if h[k] is None else torch.from_numpy(h[k]).to(dev)
    if kind == "map":
        s["g"] = _stored_potentials(h, dev)
    s["ws"] = native.Workspace(case["n"], case["m"], case["d"], case.get("precision", "fp32"))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        s["plan"].run()
        res = s["plan"].collect()
        return {k: torch.cat([r[k].reshape(-1) for r in res]) for k in ("x_out", "g_all", "f_last")}
    x, y, a, b, ws = s["x"], s["y"], s["a"], s["b"], s["ws"]
    if kind == "map":
        return dict(out=native.entropic_map_apply(x, y, s["g"], s["eps"], s["alpha"], precision=case["precision"],
                                                  workspace=ws))
    if kind == "sinkhorn":
        r = native.sinkhorn_potentials(x, y, s["eps"][0], 0.0, case["iters"], a, b, precision=case["precision"],
                                       workspace=ws)
        return dict(f=r.f, g=r.g)
    if kind == "coupling":
        eps = s["eps"][0]
        r = native.sinkhorn_potentials(x, y, eps, 0.0, case["iters"], precision=case["precision"], workspace=ws)
        met = native.coupling_metrics(x, y, r.f, r.g, eps, workspace=ws)
        row, col, _ = native.coupling_marginals(x, y, r.f, r.g, eps, workspace=ws)
        return dict(f=r.f, g=r.g, row=row, col=col, cost=met["transport_cost"], entropy=met["entropy"],
                    dual=met["dual"], mass=met["mass"])
    if kind == "pnorm":
        r, _ = native.progot_solve_pnorm(x, y, case["p"], s["alpha"], s["tau"], eps=s["eps"], max_iter=case["iters"],
                                         workspace=ws)
    else:
        r = native.progot_solve(x, y, s["alpha"], s["eps"], s["tau"], case["iters"], a, b,
                                precision=case["precision"], workspace=ws)
    return dict(x_out=r.x_out, g_all=r.g_all, f_last=r.f_last)


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    if case["kind"] == "batch":
        each = [work(dict(case, kind="progot", n=n, m=m, d=d)) for n, m, d in _batch_sizes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    kind, n, m, d = case["kind"], case["n"], case["m"], case["d"]
    pairs = float(n) * m
    K = case.get("K", 1)
    sweep, disp = 2.0 * d * pairs, 4.0 * d * pairs
    data = 4.0 * (n + m) * d
    updates = 2 * case.get("iters", 0) + 1
    if kind == "map":
        flops, nbytes = K * disp, data + 4.0 * (K * m + n * d)
    elif kind == "sinkhorn":
        flops, nbytes = updates * sweep, data + 4.0 * (n + m)
    elif kind == "coupling":
        flops, nbytes = (updates + 2) * sweep, data + 8.0 * (n + m)
    else:
        flops, nbytes = K * (updates * sweep + disp), data + 4.0 * (K * m + n * d + n)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- float64 restatement
def _sq_cost(x, y):
    c = x.mean(0)
    x, y = x - c, y - c
    return (x * x).sum(1)[:, None] + (y * y).sum(1)[None, :] - 2.0 * (x @ y.T)


def _p_cost(x, y, p):
    C = torch.zeros(len(x), len(y), dtype=x.dtype, device=x.device)
    for k in range(x.shape[1]):
        C += (x[:, k, None] - y[None, :, k]).abs_().pow_(p)
    return C / p


def _sinkhorn64(C, eps, iters, g, loga, logb):
    f = None
    for _ in range(iters):
        f = eps * (loga - torch.logsumexp((g[None, :] - C) / eps, 1))
        g = eps * (logb - torch.logsumexp((f[:, None] - C) / eps, 0))
    return f, g


def _moved64(x, y, C, g, eps, alpha, p):
    P = torch.softmax((g[None, :] - C) / eps, 1)
    if p is None:
        return x + alpha * (P @ y - x)
    z = torch.empty_like(x)
    for k in range(x.shape[1]):
        diff = x[:, k, None] - y[None, :, k]
        z[:, k] = (P * (diff.sign() * diff.abs().pow(p - 1.0))).sum(1)
    return x - alpha * z.sign() * z.abs().pow(1.0 / (p - 1.0))


def _progot64(h, iters, dev, p=None):
    x, y = (torch.from_numpy(h[k]).to(dev).double() for k in ("x", "y"))
    n, m = len(x), len(y)
    loga = torch.full((n,), -math.log(n), dtype=torch.float64, device=dev) if h["a"] is None else \
        torch.from_numpy(h["a"]).to(dev).double().log()
    logb = torch.full((m,), -math.log(m), dtype=torch.float64, device=dev) if h["b"] is None else \
        torch.from_numpy(h["b"]).to(dev).double().log()
    g = torch.zeros(m, dtype=torch.float64, device=dev)
    g_all, f = [], None
    for k, (eps, alpha) in enumerate(zip(h["eps"], h["alpha"])):
        C = _sq_cost(x, y) if p is None else _p_cost(x, y, p)
        g = g * (1.0 - alpha) if k else g
        f, g = _sinkhorn64(C, eps, iters, g, loga, logb)
        g_all.append(g)
        x = _moved64(x, y, C, g, eps, alpha, p)
    return dict(x_out=x, g_all=torch.stack(g_all), f_last=f)


def exact(case, seed):
    dev = _device()
    kind = case["kind"]
    if kind == "batch":
        res = [_progot64(h, case["iters"], dev) for h in _batch_inputs(case, seed)]
        return {k: torch.cat([r[k].reshape(-1) for r in res]) for k in ("x_out", "g_all", "f_last")}
    h = _host_inputs(case, seed)
    if kind in ("progot", "pnorm"):
        return _progot64(h, case["iters"], dev, case.get("p"))
    x, y = (torch.from_numpy(h[k]).to(dev).double() for k in ("x", "y"))
    if kind == "map":
        for g, eps, alpha in zip(_stored_potentials(h, dev).double(), h["eps"], h["alpha"]):
            x = _moved64(x, y, _sq_cost(x, y), g, eps, alpha, None)
        return dict(out=x)
    n, m, eps = len(x), len(y), h["eps"][0]
    C = _sq_cost(x, y)
    loga = torch.full((n,), -math.log(n), dtype=torch.float64, device=dev) if h["a"] is None else \
        torch.from_numpy(h["a"]).to(dev).double().log()
    logb = torch.full((m,), -math.log(m), dtype=torch.float64, device=dev) if h["b"] is None else \
        torch.from_numpy(h["b"]).to(dev).double().log()
    f, g = _sinkhorn64(C, eps, case["iters"], torch.zeros(m, dtype=torch.float64, device=dev), loga, logb)
    if kind == "sinkhorn":
        return dict(f=f, g=g)
    logP = (f[:, None] + g[None, :] - C) / eps
    P = logP.exp()
    return dict(f=f, g=g, row=P.sum(1), col=P.sum(0), cost=float((P * C).sum()), entropy=float((P - P * logP).sum()),
                dual=float(f.mean() + g.mean() - eps * P.sum()), mass=float(P.sum()))
