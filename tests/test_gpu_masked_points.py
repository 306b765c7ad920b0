"""Points masked out of a coupling by a potential of the type's lowest value: they carry nothing,
and whole tiles of them leave the metrics of the others as they are.

Tolerance: as in test_gpu_grid.py, a score (|t| <= 4 T / ln 2 + 32, T = max |x~|^2 / eps) is rounded
a few times by 2^-23; every sum of P, and of P log P per unit of log P, is off by that relative."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_05061_gb300 import native as nat  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


@pytest.mark.parametrize("scale", [0.1, 1e-3, 1e-5])
@pytest.mark.parametrize("n,m,masked", [(300, 400, slice(0, 64)), (700, 1500, slice(0, 1024)),
                                        (300, 2300, slice(256, 2176)), (200, 500, slice(64, 128))])
def test_metrics_beside_masked_targets(n, m, masked, scale):
    d = 16
    rng = np.random.default_rng(m)
    x, y = rng.standard_normal((n, d)).astype(np.float32), rng.standard_normal((m, d)).astype(np.float32)
    eps = scale * 2 * d
    C = ((x.astype(np.float64)[:, None] - y.astype(np.float64)[None]) ** 2).sum(-1)
    keep = np.ones(m, bool)
    keep[masked] = False
    b = keep / keep.sum()
    t = -C[:, keep] / eps
    mx = t.max(1, keepdims=True)
    f = (-eps * (np.log(np.exp(t - mx).sum(1)) + mx[:, 0]) - eps * np.log(n)).astype(np.float32)
    g = np.where(keep, 0.0, np.finfo(np.float32).min).astype(np.float32)
    logp = (f.astype(np.float64)[:, None] - C[:, keep]) / eps
    P = np.exp(logp)
    met = nat.coupling_metrics(dev(x), dev(y), dev(f), dev(g), eps, b=dev(b))
    r2 = max((x.astype(np.float64) ** 2).sum(1).max(), (y.astype(np.float64) ** 2).sum(1).max())
    tol = 2.0 ** -21 * (4.0 * 1.2 * r2 / eps + 16.0)
    cost, ent = float((P * C[:, keep]).sum()), float((P - P * logp).sum())
    assert abs(met["mass"] - P.sum()) <= tol * P.sum()
    assert abs(met["transport_cost"] - cost) <= tol * (cost + 2 * r2) + 2 * eps * tol * 40
    assert abs(met["entropy"] - ent) <= tol * np.abs(P - P * logp).sum() + tol * P.sum()
    row, col, _ = nat.coupling_marginals(dev(x), dev(y), dev(f), dev(g), eps, b=dev(b))
    assert float(col.cpu().numpy()[~keep].max()) == 0.0
    np.testing.assert_allclose(row.cpu().numpy(), P.sum(1), rtol=tol)
    for value in (-1e38, -1e35, -1e30, -1e22):
        g[~keep] = value
        r2, _, _ = nat.coupling_marginals(dev(x), dev(y), dev(f), dev(g), eps, b=dev(b))
        np.testing.assert_allclose(r2.cpu().numpy(), P.sum(1), rtol=tol)


@pytest.mark.parametrize("value", [np.finfo(np.float32).min, -1e36, -np.inf])
@pytest.mark.parametrize("n,m,d,K", [(777, 901, 192, 2), (2500, 2400, 64, 8)])
def test_map_beside_masked_targets(n, m, d, K, value):
    rng = np.random.default_rng(d)
    x, y = rng.standard_normal((n, d)).astype(np.float32), rng.standard_normal((m, d)).astype(np.float32)
    eps = 0.1 * 2 * d
    g = (rng.standard_normal((K, m)) * eps).astype(np.float32)
    keep = np.ones(m, bool)
    keep[64:192] = keep[300] = False
    g[:, ~keep] = value
    alpha = [1.0 / (K - k) for k in range(K)]
    out = nat.entropic_map_apply(dev(x), dev(y), dev(g), [eps] * K, alpha).cpu().numpy()
    rows = np.r_[0:20, n - 20:n]
    ref, yk = x[rows].astype(np.float64), y[keep].astype(np.float64)
    for gk, al in zip(g[:, keep].astype(np.float64), alpha):
        t = (gk - ((ref ** 2).sum(1)[:, None] + (yk ** 2).sum(1) - 2 * ref @ yk.T)) / eps
        p = np.exp(t - t.max(1, keepdims=True))
        ref = ref + al * (p @ yk / p.sum(1, keepdims=True) - ref)
    r2 = (y.astype(np.float64) ** 2).sum(1).max()
    np.testing.assert_allclose(out[rows], ref, rtol=0, atol=K * 2.0 ** -21 * (4 * r2 / eps + 16) * r2 ** 0.5)


@pytest.mark.parametrize("value", [np.finfo(np.float32).min, -1e36, -np.inf])
@pytest.mark.parametrize("n,m", [(300, 500), (128, 64), (200, 190)])
def test_loop_from_a_masked_start(n, m, value):
    """One f-update from a given g; half a tile of it masked, and a tile and a half."""
    d = 16
    rng = np.random.default_rng(n)
    x, y = rng.standard_normal((n, d)).astype(np.float32), rng.standard_normal((m, d)).astype(np.float32)
    eps = 0.1 * 2 * d
    C = ((x.astype(np.float64)[:, None] - y.astype(np.float64)[None]) ** 2).sum(-1)
    for masked in (slice(0, 63), slice(64, m - 1), slice(0, m - 1)):
        keep = np.ones(m, bool)
        keep[masked] = False
        g = np.where(keep, 0.0, value).astype(np.float32)
        t = -C[:, keep] / eps
        mx = t.max(1, keepdims=True)
        f = -eps * (np.log(np.exp(t - mx).sum(1)) + mx[:, 0]) - eps * np.log(n)
        r = nat.sinkhorn_potentials(dev(x), dev(y), eps, 0.0, 1, f=dev(np.zeros(n)), g=dev(g))
        r2 = max((x.astype(np.float64) ** 2).sum(1).max(), (y.astype(np.float64) ** 2).sum(1).max())
        np.testing.assert_allclose(r.f.cpu().numpy(), f, rtol=0, atol=eps * 2.0 ** -21 * (4 * 1.2 * r2 / eps + 16))
        assert bool(torch.isfinite(r.g).all())


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("n,m,d,j", [(200, 500, 16, 70), (200, 500, 16, 133), (1500, 2500, 16, 3), (1500, 2500, 16, 2311),
                                     (900, 700, 64, 650)])
def test_potentials_that_are_not_finite_show(n, m, d, j, value):
    """One NaN (or infinite) g_j belongs to every row sum."""
    rng = np.random.default_rng(j)
    x, y = rng.standard_normal((n, d)), rng.standard_normal((m, d))
    f, g = np.zeros(n), np.zeros(m)
    g[j] = value
    eps = 0.2 * d
    row, _, err = nat.coupling_marginals(dev(x), dev(y), dev(f), dev(g), eps)
    assert not bool(torch.isfinite(row).any()) and not np.isfinite(err)
    _, col, err = nat.coupling_marginals(dev(y), dev(x), dev(g), dev(f), eps)
    assert not bool(torch.isfinite(col).any()) and not np.isfinite(err)
    with pytest.raises(nat.ProgOTError) as ei:
        nat.sinkhorn_potentials(dev(x), dev(y), eps, 0.0, 3, f=dev(f), g=dev(g))
    assert ei.value.code == nat.PROGOT_ERR_NUMERIC
