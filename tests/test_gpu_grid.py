"""Integer-grid operands of the float32 path (csrc/grid_split.cuh): sweeps, loops and map
steps against the float64 oracle at the edges of their tiles, K steps and parts, and on
clouds that stress the split (outliers, clouds of unequal size, tiny and huge eps).

Tolerances: with T = max |x~|^2 / eps (natural log units; x~ centred) the sweeps round t_ij
once (2^-24 |t|, |t| <= 4 T / ln 2 + 32), the potentials once more, and sums and exponentials
add a few 2^-23; a bound of 2^-21 (4 T + 16) covers all of it for a marginal, and a map step
moves a point by at most that times the spread of the targets."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import progot_oracle as O  # noqa: E402
from paper_2406_05061_gb300 import native as nat  # noqa: E402
from paper_2406_05061_gb300 import workloads as W  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def clouds(n, m, d, seed, kind="gmm"):
    if kind == "gmm":
        p = W.gmm_pair(n, m, d, seed=seed, k=3)
        return p.x, p.y
    rng = np.random.default_rng(seed)
    x, y = rng.standard_normal((n, d)), rng.standard_normal((m, d))
    if kind == "outlier":
        x[0] *= 300.0
    elif kind == "unequal":
        y *= 1e-3
    elif kind == "far":
        x, y = x + 100.0, y + 100.0
    return x.astype(np.float32), y.astype(np.float32)


def sq_cost(x, y):
    x, y = x.astype(np.float64), y.astype(np.float64)
    return ((x[:, None, :] - y[None, :, :]) ** 2).sum(-1)


def bound(x, y, eps):
    mu = 0.5 * (x.astype(np.float64).mean(0) + y.astype(np.float64).mean(0))
    r2 = max(((x - mu) ** 2).sum(1).max(), ((y - mu) ** 2).sum(1).max())
    return 2.0 ** -21 * (4.0 * r2 / eps + 16.0)


@pytest.mark.parametrize("n,m,d,kind", [(1, 1, 1, "gmm"), (127, 129, 15, "gmm"), (128, 256, 16, "gmm"),
                                        (257, 128, 17, "gmm"), (300, 520, 48, "gmm"), (129, 383, 49, "gmm"),
                                        (1000, 700, 64, "gmm"), (200, 300, 65, "gmm"), (130, 500, 256, "gmm"),
                                        (140, 260, 400, "gmm"), (300, 200, 8, "outlier"), (300, 200, 8, "unequal"),
                                        (300, 200, 8, "far")])
def test_grid_marginals_against_float64(n, m, d, kind):
    x, y = clouds(n, m, d, seed=n + d, kind=kind)
    C = sq_cost(x, y)
    eps = 0.05 * float(np.median(C)) + 1e-3
    f = np.zeros(n)
    g = -eps * np.log(np.exp(-(C - C.min(0)) / eps).sum(0)) + C.min(0) - eps * np.log(m)
    f, g = f.astype(np.float32), g.astype(np.float32)
    P = np.exp((f[:, None].astype(np.float64) + g[None, :] - C) / eps)
    row, col, _ = nat.coupling_marginals(dev(x), dev(y), dev(f), dev(g), eps)
    tol = bound(x, y, eps)
    np.testing.assert_allclose(row.cpu().numpy(), P.sum(1), rtol=tol, atol=tol * P.sum(1).max() * 2.0 ** -20)
    np.testing.assert_allclose(col.cpu().numpy(), P.sum(0), rtol=tol)


@pytest.mark.parametrize("n,m,d", [(5, 2, 1), (128, 128, 16), (129, 257, 17), (300, 260, 33), (640, 385, 48),
                                   (257, 640, 49), (500, 900, 64)])
def test_grid_loop_against_float64(n, m, d):
    x, y = clouds(n, m, d, seed=d)
    C = sq_cost(x, y)
    eps = 0.05 * float(C.mean())
    rng = np.random.default_rng(d)
    a = rng.uniform(0.5, 1.5, n).astype(np.float32)
    b = rng.uniform(0.5, 1.5, m).astype(np.float32)
    a, b = a / a.sum(), b / b.sum()
    its = 7  # odd: f and the bias rows of g end in their second buffers
    f, g = np.zeros(n), np.zeros(m)
    for _ in range(its):
        f = eps * np.log(a.astype(np.float64)) + O.softmin(C - g[None, :], eps)
        g = eps * np.log(b.astype(np.float64)) + O.softmin((C - f[:, None]).T, eps)
    r = nat.sinkhorn_potentials(dev(x), dev(y), eps, 0.0, its, dev(a), dev(b))
    assert r.iters == its and r.status == nat.PROGOT_ERR_NOT_CONVERGED
    tol = eps * bound(x, y, eps) * 2 * its
    np.testing.assert_allclose(r.f.cpu().numpy(), f, rtol=0, atol=tol)
    np.testing.assert_allclose(r.g.cpu().numpy(), g, rtol=0, atol=tol)


@pytest.mark.parametrize("n,m,d,precision", [(700, 640, 64, "fp32"), (2000, 127, 128, "fp32"), (130, 4000, 65, "fp32"),
                                             (4100, 513, 16, "fp32"), (1500, 1500, 300, "fp32"),
                                             (257, 300, 257, "bf16x3"), (128, 129, 700, "bf16x3"),
                                             (1, 64, 320, "bf16x3")])
def test_grid_map_against_float64(n, m, d, precision):
    """Cluster splits, several coordinate chunks, ragged rows, columns and coordinates; two
    steps, so that the second runs on the moved cloud (float32: the hull's exponents)."""
    x, y = clouds(n, m, d, seed=m)
    C = sq_cost(x[:min(n, 400)], y)
    eps = 0.1 * float(C.mean())
    rng = np.random.default_rng(n)
    gs = (rng.standard_normal((2, m)) * eps).astype(np.float32)
    out = nat.entropic_map_apply(dev(x), dev(y), dev(gs), [2 * eps, eps], [0.5, 1.0], precision=precision)
    rows = np.unique(np.r_[0, n - 1, rng.integers(0, n, 60)])
    ref = x[rows].astype(np.float64)
    for g, e, al in zip(gs, (2 * eps, eps), (0.5, 1.0)):
        t = (g[None, :].astype(np.float64) - sq_cost(ref, y)) / e
        p = np.exp(t - t.max(1, keepdims=True))
        ref = ref + al * (p @ y.astype(np.float64) / p.sum(1, keepdims=True) - ref)
    spread = np.sqrt(((y - y.mean(0)) ** 2).sum(1).max())
    # two parts (bf16x3): the operands carry 2^-25 of the largest norm per coordinate
    tol = bound(x, y, eps) * spread * (1 if precision == "fp32" else 8)
    np.testing.assert_allclose(out.cpu().numpy()[rows], ref, rtol=0, atol=tol)


def test_float32_workspace_without_grid_operands_still_serves():
    """A workspace of the size the CUDA-core path needs is accepted and gives its results."""
    x, y = clouds(300, 260, 16, seed=3)
    eps, its = 20.0, 20
    full = nat.sinkhorn_potentials(dev(x), dev(y), eps, 0.0, its)
    big = nat.workspace_size(300, 260, 16)
    parts = 6 * 300 * 64 * 2  # at least the operands' bytes less
    size = big - parts
    buf = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
    ptr = (buf.data_ptr() + 255) & ~255
    f = torch.zeros(300, device="cuda")
    g = torch.zeros(260, device="cuda")
    it, err = ctypes.c_int32(0), ctypes.c_double(0.0)
    xd, yd = dev(x), dev(y)
    rc = nat.lib().sinkhorn_potentials(ctypes.c_void_p(xd.data_ptr()), None, 300, ctypes.c_void_p(yd.data_ptr()), None,
                                       260, 16, eps, 0.0, its, 0, ctypes.c_void_p(f.data_ptr()),
                                       ctypes.c_void_p(g.data_ptr()), 1, ctypes.byref(it), ctypes.byref(err),
                                       ctypes.c_void_p(ptr), size, None)
    torch.cuda.synchronize()
    assert rc == nat.PROGOT_ERR_NOT_CONVERGED and it.value == its
    tol = 2 * its * eps * bound(x, y, eps) + 2.0 ** -21 * float((x ** 2).sum(1).max() + (y ** 2).sum(1).max())
    np.testing.assert_allclose(f.cpu().numpy(), full.f.cpu().numpy(), rtol=0, atol=tol)
    np.testing.assert_allclose(g.cpu().numpy(), full.g.cpu().numpy(), rtol=0, atol=tol)


def test_grid_zero_weight_points_carry_no_mass():
    x, y = clouds(200, 300, 16, seed=9)
    b = np.full(300, 1.0 / 299, np.float32)
    b[17] = 0.0
    r = nat.sinkhorn_potentials(dev(x), dev(y), 30.0, 1e-4, 500, b=dev(b))
    assert r.status == nat.PROGOT_OK
    g = r.g.cpu().numpy()
    assert g[17] == -np.inf and np.isfinite(np.delete(g, 17)).all() and np.isfinite(r.f.cpu().numpy()).all()
