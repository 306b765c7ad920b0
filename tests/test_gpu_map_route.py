"""Which kernels a float32 map runs on, and that both routes give the float64 result.

Tolerance of the values: as in test_gpu_grid.py, a step rounds t_ij (|t| <= 4 T / ln 2 + 32,
T = max |x~|^2 / eps) and its sums by a few 2^-23, which moves a point by at most that times the
spread of the targets; K steps add up."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_05061_gb300 import native as nat  # noqa: E402
from paper_2406_05061_gb300 import workloads as W  # noqa: E402

CUDA_CORES = 2  # launches a step: log-sum-exp and map (the target's norms once besides)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def run(n, m, d, K, rows=40):
    p = W.gmm_pair(n, m, d, seed=n + d, k=3) if d <= 64 else W.sphere_mixture_pair(n, m, d, seed=n + d)
    x, y = p.x, p.y
    mu = 0.5 * (x.astype(np.float64).mean(0) + y.astype(np.float64).mean(0))
    r2 = max(((x - mu) ** 2).sum(1).max(), ((y - mu) ** 2).sum(1).max())
    eps = [0.1 * r2 * (2.0 - k / K) for k in range(K)]
    alpha = [1.0 / (K - k) for k in range(K)]
    rng = np.random.default_rng(n)
    g = (rng.standard_normal((K, m)) * eps[-1]).astype(np.float32)
    args = (dev(x), dev(y), dev(g), eps, alpha)
    ws = nat.Workspace(n, m, d)
    nat.launch_count(reset=True)
    out = nat.entropic_map_apply(*args, workspace=ws).cpu().numpy()
    launches = nat.launch_count(reset=True)
    idx = np.unique(np.r_[0, n - 1, rng.integers(0, n, rows)])
    ref, y64 = x[idx].astype(np.float64), y.astype(np.float64)
    for gk, e, al in zip(g.astype(np.float64), eps, alpha):
        c = (ref ** 2).sum(1)[:, None] + (y64 ** 2).sum(1) - 2 * ref @ y64.T
        t = (gk - c) / e
        w = np.exp(t - t.max(1, keepdims=True))
        ref = ref + al * (w @ y64 / w.sum(1, keepdims=True) - ref)
    tol = K * 2.0 ** -21 * (4.0 * r2 / eps[-1] + 16.0) * np.sqrt(((y - y.mean(0)) ** 2).sum(1).max())
    np.testing.assert_allclose(out[idx], ref, rtol=0, atol=tol)
    return launches


@pytest.mark.parametrize("n,m,d,K", [(1000, 2048, 3, 1), (1500, 1500, 16, 1), (700, 700, 32, 1), (500, 500, 16, 2),
                                     (128, 20000, 2, 3), (1000, 1000, 16, 4), (300, 300, 2, 8)])
def test_short_and_small_float32_maps_stay_on_cuda_cores(n, m, d, K):
    assert run(n, m, d, K) == CUDA_CORES * K + 1


@pytest.mark.parametrize("n,m,d,K", [(6000, 5777, 3, 1), (3000, 3000, 8, 1), (500, 500, 100, 1), (1000, 1000, 64, 2),
                                     (4099, 4300, 16, 4), (3001, 3070, 48, 3), (129, 383, 130, 8), (130, 500, 80, 16),
                                     (2001, 127, 250, 2), (1, 640, 256, 6), (777, 901, 192, 2)])
def test_float32_maps_on_the_tensor_cores(n, m, d, K):
    assert run(n, m, d, K) > CUDA_CORES * K + 1
