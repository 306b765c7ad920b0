"""The map step beyond d = 256 at the mixed precisions: the step's own operands are the integer
grid's, whatever the precision of the loop, so a map with given potentials is a float32 result.

Tolerance: as in test_gpu_grid.py, t_ij (|t| <= 4 T / ln 2 + 32, T = max |x~|^2 / eps) and the
sums are rounded a few times by 2^-23, which moves a point by at most that times the spread of
the targets; above 0.5 spreads the bound says nothing and only finiteness is asked for."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_05061_gb300 import native as nat  # noqa: E402
from paper_2406_05061_gb300 import workloads as W  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def sq_cost(x, y):
    x, y = x.astype(np.float64), y.astype(np.float64)
    return (x * x).sum(1)[:, None] + (y * y).sum(1) - 2.0 * x @ y.T


def fitted_potential(x, y, eps):
    """g after four float64 updates."""
    C = sq_cost(x, y)

    def softmin(z, axis):
        lo = z.min(axis, keepdims=True)
        return (lo - eps * np.log(np.exp(-(z - lo) / eps).sum(axis, keepdims=True))).squeeze(axis)

    g = np.zeros(len(y))
    for _ in range(4):
        f = softmin(C - g[None, :], 1)
        g = softmin(C - f[:, None], 0)
    return g.astype(np.float32)


def exact_map(x, y, g, eps):
    t = (g[None, :].astype(np.float64) - sq_cost(x, y)) / eps
    p = np.exp(t - t.max(1, keepdims=True))
    return p @ y.astype(np.float64) / p.sum(1, keepdims=True)


def bound(x, y, eps):
    mu = 0.5 * (x.astype(np.float64).mean(0) + y.astype(np.float64).mean(0))
    r2 = max(((x - mu) ** 2).sum(1).max(), ((y - mu) ** 2).sum(1).max())
    return 2.0 ** -21 * (4.0 * r2 / eps + 16.0)


@pytest.mark.parametrize("precision,scale", [("bf16", 0.02), ("bf16", 3e-3), ("bf16", 1e-3), ("bf16", 1e-5),
                                             ("bf16x3", 1e-3), ("bf16x3", 1e-5)])
@pytest.mark.parametrize("n,m,d,cloud", [(800, 800, 300, "sphere"), (800, 700, 400, "gmm"), (333, 257, 1000, "gmm")])
def test_map_far_below_the_cost_stays_finite(n, m, d, cloud, precision, scale):
    """eps = scale * mean cost / 20: the loop's bf16 products are off by whole bits of t there."""
    p = W.gmm_pair(n, m, d, seed=3) if cloud == "gmm" else W.sphere_mixture_pair(n, m, d, seed=3)
    x, y = p.x, p.y
    eps = scale * float(sq_cost(x, y).mean()) / 20.0
    g = fitted_potential(x, y, eps)
    out = nat.entropic_map_apply(dev(x), dev(y), dev(g[None]), [eps], [1.0], precision=precision).cpu().numpy()
    assert np.isfinite(out).all()
    spread = np.sqrt(((y - y.mean(0)) ** 2).sum(1).max())
    tol = 8 * bound(x, y, eps)
    if tol < 0.5:
        np.testing.assert_allclose(out, exact_map(x, y, g, eps), rtol=0, atol=tol * spread)


@pytest.mark.parametrize("d,far", [(300, 1.0), (300, 16.0), (1000, 1.0), (1000, 16.0), (1024, 4.0), (300, 300.0),
                                   (1000, 100.0), (3000, 40.0), (3000, 1000.0)])
@pytest.mark.parametrize("precision", ["bf16x3", "bf16", "fp32"])
def test_map_is_no_further_from_float64_than_float32_products(d, far, precision):
    """The CUDA-core map (float32 throughout) is the measure; a quarter on top for the sample."""
    rng = np.random.default_rng(d)
    x, y = rng.standard_normal((1500, d)), rng.standard_normal((1400, d))
    y[0] *= far
    x, y = x.astype(np.float32), y.astype(np.float32)
    eps = 0.1 * d
    g = (rng.standard_normal(1400) * eps).astype(np.float32)
    if far > 1:
        g[0] = -1e9 * eps  # without weight: its own score is no float32 result
    ref = exact_map(x, y, g, eps)
    args = (dev(x), dev(y), dev(g[None]), [eps], [1.0])
    err = {}
    for tc in (True, False):
        nat.set_map_tc(tc)
        try:
            out = nat.entropic_map_apply(*args, precision=precision if tc else "bf16x3")
        finally:
            nat.set_map_tc(True)
        err[tc] = float(np.sqrt(((out.cpu().numpy() - ref) ** 2).mean()))
    assert err[True] <= 1.25 * err[False], err
