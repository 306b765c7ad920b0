"""Float32 entropic maps on the tensor cores: a bounded wait that runs out is reported, and a
captured map (which cannot read that report back) runs where nothing waits."""
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


def test_expired_wait_of_a_float32_map_is_reported():
    args = problem()
    nat.test_withhold_initial_betas(True)
    try:
        with pytest.raises(nat.ProgOTError) as ei:
            nat.entropic_map_apply(*args)
        assert ei.value.code == nat.PROGOT_ERR_TIMEOUT
    finally:
        nat.test_withhold_initial_betas(False)
    assert bool(torch.isfinite(nat.entropic_map_apply(*args)).all())


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
    # two float32 evaluations of t (|t| up to 4 |x~|^2 / eps) and two steps
    r2 = float((y - y.mean(0)).pow(2).sum(1).max())
    tol = 2 * 2 * 2.0 ** -21 * (4 * r2 / eps[1] + 16) * r2 ** 0.5
    assert float((out - ref).abs().max()) <= tol
