"""Float32 entropic maps on the tensor cores do not wait for the device: steps that a bounded wait
cost are done again behind them, in a captured map too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_05061_gb300 import native as nat  # noqa: E402
from paper_2406_05061_gb300 import workloads as W  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def problem():
    p = W.gmm_pair(2500, 2300, 64, seed=2, k=3)
    eps = 0.2 * float(np.mean((p.x - p.y[: len(p.x)].mean(0)) ** 2) * 64)
    g = np.random.default_rng(0).standard_normal((2, 2300)).astype(np.float32) * np.float32(eps)
    return dev(p.x), dev(p.y), dev(g), [2 * eps, eps], [0.5, 1.0]


def tolerance(x, y, eps, steps):
    """Two float32 evaluations of t (|t| up to 4 |x~|^2 / eps) and their steps."""
    r2 = float((y - y.mean(0)).pow(2).sum(1).max())
    return 2 * steps * 2.0 ** -21 * (4 * r2 / eps + 16) * r2 ** 0.5


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("K", [2, 35])
def test_expired_wait_of_a_float32_map_is_made_good(in_place, K):
    x, y, g, eps, _ = problem()
    g, eps = g[:1].repeat(K, 1), [eps[0]] * K
    alpha = [1.0 / (K - k) for k in range(K)]
    ref = nat.entropic_map_apply(x, y, g, eps, alpha)
    nat.test_withhold_initial_betas(True)
    try:
        xq = x.clone()
        out = nat.entropic_map_apply(xq, y, g, eps, alpha, out=xq if in_place else None)
    finally:
        nat.test_withhold_initial_betas(False)
    assert float((out - ref).abs().max()) <= tolerance(x, y, eps[0], K)
    assert not torch.equal(out, ref)  # by other kernels


def test_captured_float32_map_replays_on_new_points():
    x, y, g, eps, alpha = problem()
    ws = nat.Workspace(2500, 2300, 64)
    out = torch.empty_like(x)
    nat.entropic_map_apply(x, y, g, eps, alpha, out=out, workspace=ws)  # kernels are loaded
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        nat.entropic_map_apply(x, y, g, eps, alpha, out=out, workspace=ws)
    x.copy_(x.flip(0))
    graph.replay()
    torch.cuda.synchronize()
    ref = nat.entropic_map_apply(x, y, g, eps, alpha, workspace=ws)
    assert float((out - ref).abs().max()) <= tolerance(x, y, eps[1], 2)


def test_captured_float32_map_of_far_points():
    """Which kernels run is decided on the device: a replay on other clouds takes its own way."""
    x, y, g, eps, alpha = problem()
    ws = nat.Workspace(2500, 2300, 64)
    out = torch.empty_like(x)
    nat.entropic_map_apply(x, y, g, eps, alpha, out=out, workspace=ws)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        nat.entropic_map_apply(x, y, g, eps, alpha, out=out, workspace=ws)
    graph.replay()
    torch.cuda.synchronize()
    near = out.clone()
    x[0] *= 3e5  # a far query: the other rows' paths are their own
    graph.replay()
    torch.cuda.synchronize()
    assert float((out[1:] - near[1:]).abs().max()) <= tolerance(x, y, eps[1], 2)


def test_float32_map_returns_before_the_device_is_done():
    x, y, g, eps, alpha = problem()
    ws = nat.Workspace(2500, 2300, 64)
    out = torch.empty_like(x)
    nat.entropic_map_apply(x, y, g, eps, alpha, out=out, workspace=ws)
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    torch.cuda._sleep(200_000_000)  # about 0.1 s of the stream's time
    nat.entropic_map_apply(x, y, g, eps, alpha, out=out, workspace=ws)
    done.record()
    assert not done.query()
    torch.cuda.synchronize()
