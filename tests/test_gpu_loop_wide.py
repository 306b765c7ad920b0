"""The persistent loop with A's row block in TMEM (128 < d <= 256, 64 column tiles a CTA or more: from
about 12,600 points on) against float64.

Tolerance: two iterations of four updates, each off by eps times the error of t. bf16x3 omits terms of
3 2^-18 |x~||y~| c and truncates sums of 3 d / 16 steps at 2^-23; hi parts alone are off by 2^-8 |x~||y~| c;
c = 2 / eps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_05061_gb300 import native as nat  # noqa: E402


@pytest.mark.parametrize("n,m,d,precision", [(12901, 12700, 256, "bf16x3"), (12700, 12999, 130, "bf16x3"),
                                             (13000, 12650, 192, "bf16"), (25000, 6500, 200, "bf16x3")])
def test_loop_of_many_tiles(n, m, d, precision):
    gen = torch.Generator(device="cuda").manual_seed(d)
    x = torch.randn(n, d, device="cuda", generator=gen)
    y = torch.randn(m, d, device="cuda", generator=gen) + 0.1
    eps, its = 0.2 * d, 2
    x64, y64 = x.double(), y.double()
    C = (x64 * x64).sum(1)[:, None] + (y64 * y64).sum(1)[None] - 2.0 * x64 @ y64.T
    g = torch.zeros(m, dtype=torch.float64, device="cuda")
    for _ in range(its):
        f = -eps * torch.logsumexp((g[None, :] - C) / eps, 1) - eps * np.log(n)
        g = -eps * torch.logsumexp((f[:, None] - C) / eps, 0) - eps * np.log(m)
    r = nat.sinkhorn_potentials(x, y, eps, 0.0, its, precision=precision)
    assert r.iters == its
    rel = 3 * 2.0 ** -18 + 3 * d / 16 * 2.0 ** -23 if precision == "bf16x3" else 2.0 ** -8
    scale = float(x64.norm(dim=1).max() * (y64 - 0.05).norm(dim=1).max())
    tol = 2 * its * 2 * rel * scale
    assert float((r.f - f).abs().max()) <= tol and float((r.g - g).abs().max()) <= tol
