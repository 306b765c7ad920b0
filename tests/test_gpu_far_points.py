"""Clouds with far points, rows that are not finite and eps far below the cost: what the
float32 calls return for the ordinary points stays what float32 products give.

Tolerances: a float32 evaluation of t_ij = (g_j - |x_i - y_j|^2) / eps by products has an error
of a few 2^-24 of the terms it is made of, |x_i||y_j| / eps, |y_j|^2 / eps and |g_j| / eps of that
very pair (norms about the midpoint of the clouds' typical points); a row's sum then has the mean
of its pairs' errors under its own weights, and a few 2^-23 of its own. ``pair_error`` takes
2^-21 of the terms plus 2^-20, eight roundings each."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_05061_gb300 import native as nat  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def clouds(n, m, d, seed, far_x=1.0, far_y=1.0):
    rng = np.random.default_rng(seed)
    x, y = rng.standard_normal((n, d)), rng.standard_normal((m, d))
    x[0] *= far_x
    y[0] *= far_y
    return x.astype(np.float32), y.astype(np.float32)


def sq_cost(x, y):
    x, y = x.astype(np.float64), y.astype(np.float64)
    return ((x[:, None, :] - y[None, :, :]) ** 2).sum(-1)


def pair_error(x, y, g, eps):
    xn, yn = (np.sqrt((v.astype(np.float64) ** 2).sum(1)) for v in (x, y))
    return 2.0 ** -21 * (2 * xn[:, None] * yn + xn[:, None] ** 2 + yn ** 2 + np.abs(g)) / eps + 2.0 ** -20


def far_potential(x, y, eps):
    """g of a column-feasible plan against x without its far point: the far y has its own weight."""
    C = sq_cost(x, y)[1:]
    t = -C / eps
    m = t.max(0)
    return (-eps * (np.log(np.exp(t - m).sum(0)) + m) - eps * np.log(y.shape[0])).astype(np.float32)


def row_terms(x, y, g, eps):
    """Weights of every row's pairs (float64) and the row's log-sum-exp."""
    t = (g[None, :].astype(np.float64) - sq_cost(x, y)) / eps
    mx = t.max(1, keepdims=True)
    p = np.exp(t - mx)
    return p / p.sum(1, keepdims=True), np.log(p.sum(1)) + mx[:, 0]


@pytest.mark.parametrize("far_x,far_y", [(3e4, 1.0), (1e5, 3e4), (1.0, 1e5)])
@pytest.mark.parametrize("n,m,d", [(5300, 5200, 24), (3500, 3049, 64)])
def test_map_of_ordinary_points_beside_very_far_ones(n, m, d, far_x, far_y):
    x, y = clouds(n, m, d, seed=d, far_x=far_x, far_y=far_y)
    eps = 0.05 * 2.0 * d
    g = far_potential(x, y, eps)
    # the far target weighs nothing: its own t is off by far more than one in float32, so that
    # whether it has a weight is not a float32 result
    g[0] -= 1e13 if far_y > 1 else 0.0
    out = nat.entropic_map_apply(dev(x), dev(y), dev(g[None]), [eps], [1.0]).cpu().numpy()
    w, _ = row_terms(x, y, g, eps)
    ref = w @ y.astype(np.float64)
    dt = pair_error(x, y, g, eps)
    # d(sum w y) = sum w (dt - mean dt) (y - ref): at most twice the weighted |dt| |y|
    yn = np.sqrt((y.astype(np.float64) ** 2).sum(1))
    tol = 2 * (w * dt * (yn[None, :] + yn.max() * 2.0 ** -22 + 1.0)).sum(1)
    err = np.abs(out - ref).max(1)
    assert (err[1:] <= tol[1:]).all(), (err[1:] / tol[1:]).max()


def test_map_rows_that_are_not_finite_stay_alone():
    n, m, d = 2500, 2300, 64
    x, y = clouds(n, m, d, seed=1)
    eps = 0.1 * 2.0 * d
    g = np.stack([far_potential(x, y, e) for e in (2 * eps, eps)])
    clean = nat.entropic_map_apply(dev(x), dev(y), dev(g), [2 * eps, eps], [0.5, 1.0]).cpu().numpy()
    for bad in (np.nan, np.inf, 1e25):
        z = x.copy()
        z[7, 3] = bad
        out = nat.entropic_map_apply(dev(z), dev(y), dev(g), [2 * eps, eps], [0.5, 1.0]).cpu().numpy()
        rest = np.arange(n) != 7
        assert np.isfinite(out[rest]).all()
        # both are float32 results of the same rows: twice two steps' errors of the ordinary pairs
        dt = float(pair_error(x, y, g[1], eps).max())
        np.testing.assert_allclose(out[rest], clean[rest], rtol=0, atol=8 * dt * np.abs(y).max())


@pytest.mark.parametrize("n,m", [(300, 200), (300, 160), (300, 250), (640, 129)])
@pytest.mark.parametrize("loop", [True, False])
def test_loop_out_of_the_grids_range_keeps_finite_potentials(n, m, loop):
    """The last tile's second half is padding only where 1 <= m mod 128 <= 64."""
    x, y = clouds(n, m, 8, seed=m, far_x=3000.0, far_y=3000.0)
    its = 4
    nat.set_loop_tc(loop)
    try:
        r = nat.sinkhorn_potentials(dev(x), dev(y), 0.5, 0.0, its)
    finally:
        nat.set_loop_tc(True)
    assert r.iters == its and r.status == nat.PROGOT_ERR_NOT_CONVERGED
    assert np.isfinite(r.err) and bool(torch.isfinite(r.f).all()) and bool(torch.isfinite(r.g).all())


def test_marginals_and_metrics_beside_very_far_points():
    x, y = clouds(500, 450, 16, seed=5, far_x=2e4, far_y=2e4)
    eps = 0.05 * 2.0 * 16
    g = far_potential(x, y, eps)
    g[0] -= 1e12  # the far points carry no mass: a float32 potential of theirs is off by whole eps
    w, lse = row_terms(x, y, g, eps)
    f = (-eps * lse - eps * np.log(500)).astype(np.float32)
    f[0] -= 1e12
    P = np.exp((f[:, None].astype(np.float64) + g[None, :] - sq_cost(x, y)) / eps)
    row, _, _ = nat.coupling_marginals(dev(x), dev(y), dev(f), dev(g), eps)
    xn = (x.astype(np.float64) ** 2).sum(1)
    tol = (w * pair_error(x, y, g, eps)).sum(1) + 2.0 ** -21 * (np.abs(f) + xn) / eps + 2.0 ** -20
    err = np.abs(row.cpu().numpy()[1:] / P.sum(1)[1:] - 1)
    assert (err <= tol[1:]).all(), (err / tol[1:]).max()
    met = nat.coupling_metrics(dev(x), dev(y), dev(f), dev(g), eps)
    assert abs(met["mass"] - P.sum()) <= (tol[1:] * P.sum(1)[1:]).sum()


@pytest.mark.parametrize("far", [100.0, 300.0, 1000.0])
@pytest.mark.parametrize("n,m,d", [(300, 300, 64), (500, 450, 16), (260, 390, 33)])
def test_far_points_in_both_clouds_leave_the_others_float32_accuracy(n, m, d, far):
    x, y = clouds(n, m, d, seed=n + d, far_x=far, far_y=far)
    eps = 0.05 * 2.0 * d
    g = far_potential(x, y, eps)
    g[0] -= 1e12  # as above
    w, lse = row_terms(x, y, g, eps)
    f = (-eps * lse - eps * np.log(n)).astype(np.float32)
    P = np.exp((f[:, None].astype(np.float64) + g[None, :] - sq_cost(x, y)) / eps)
    row, _, _ = nat.coupling_marginals(dev(x), dev(y), dev(f), dev(g), eps)
    xn = (x.astype(np.float64) ** 2).sum(1)
    dt = pair_error(x, y, g, eps)
    tol = (w * dt).sum(1) + 2.0 ** -21 * (np.abs(f) + xn) / eps + 2.0 ** -20
    err = np.abs(row.cpu().numpy()[1:] / P.sum(1)[1:] - 1)
    assert (err <= tol[1:] / 4).all(), (err / tol[1:]).max()  # two roundings a term, not eight


@pytest.mark.parametrize("far", [100.0, 300.0, 1000.0])
@pytest.mark.parametrize("n,m,d", [(300, 300, 64), (1500, 1450, 16)])
def test_one_loop_update_beside_far_points(n, m, d, far):
    """f of one iteration from g = 0 (the far column weighs nothing in the other rows)."""
    x, y = clouds(n, m, d, seed=n + 2 * d, far_x=far, far_y=far)
    eps = 0.05 * 2.0 * d
    r = nat.sinkhorn_potentials(dev(x), dev(y), eps, 0.0, 1)
    g0 = np.zeros(m, np.float32)
    w, lse = row_terms(x, y, g0, eps)
    xn = (x.astype(np.float64) ** 2).sum(1)
    tol = eps * ((w * pair_error(x, y, g0, eps)).sum(1) + 2.0 ** -21 * xn / eps + 2.0 ** -20)
    err = np.abs(r.f.cpu().numpy() - (-eps * lse - eps * np.log(n)))
    assert (err[1:] <= tol[1:] / 4).all(), (err[1:] / tol[1:]).max()


@pytest.mark.parametrize("n,m,d,K", [(2500, 2300, 64, 3), (1100, 1000, 250, 2), (777, 901, 300, 35)])
def test_map_steps_beside_very_far_queries(n, m, d, K):
    """Several steps done again by float32 FMAs: ragged rows, columns and coordinates, more steps than
    one launch takes."""
    x, y = clouds(n, m, d, seed=K, far_x=1e6)
    eps = 0.1 * 2.0 * d
    g = np.random.default_rng(d).standard_normal((K, m)).astype(np.float32) * np.float32(eps)
    alpha = [1.0 / (K - k) for k in range(K)]
    for tc in (True, False):
        nat.set_map_tc(tc)
        try:
            out = nat.entropic_map_apply(dev(x), dev(y), dev(g), [eps] * K, alpha).cpu().numpy()
        finally:
            nat.set_map_tc(True)
        rows = np.r_[1:20, n - 20:n]
        ref, y64 = x[rows].astype(np.float64), y.astype(np.float64)
        for gk, al in zip(g.astype(np.float64), alpha):
            t = (gk - ((ref ** 2).sum(1)[:, None] + (y64 ** 2).sum(1) - 2 * ref @ y64.T)) / eps
            p = np.exp(t - t.max(1, keepdims=True))
            ref = ref + al * (p @ y64 / p.sum(1, keepdims=True) - ref)
        r2 = (y64 ** 2).sum(1).max()
        np.testing.assert_allclose(out[rows], ref, rtol=0, atol=K * 2.0 ** -21 * (4 * r2 / eps + 16) * r2 ** 0.5)
