"""Loops over a kept p-norm cost are no further from float64 than loops that form it tile by tile
(a workspace one byte short of the kept cost). The errors are averaged over seeds; a tenth on top for
what the seeds leave."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_05061_gb300 import native as nat  # noqa: E402
from paper_2406_05061_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("n,m,d,p", [(773, 303, 10, 1.25), (1147, 1020, 4, 1.5), (900, 1300, 27, 1.5), (640, 513, 13, 3.0)])
def test_kept_cost_is_as_exact_as_the_cost_formed_again(n, m, d, p):
    its, err = 4, {True: [], False: []}
    for seed in range(6):
        pr = W.gmm_pair(n, m, d, seed=100 + seed, k=3)
        x, y = torch.from_numpy(pr.x).cuda(), torch.from_numpy(pr.y).cuda()
        C = (x.double()[:, None, :] - y.double()[None]).abs().pow(p).sum(-1) / p
        eps = float(C.mean()) / 20
        g = torch.zeros(m, dtype=torch.float64, device="cuda")
        for _ in range(its):
            f = -eps * torch.logsumexp((g[None, :] - C) / eps, 1) - eps * np.log(n)
            g = -eps * torch.logsumexp((f[:, None] - C) / eps, 0) - eps * np.log(m)
        for kept in (True, False):
            ws = nat.Workspace(n, m, d)
            ws.bytes -= 0 if kept else 1
            r = nat.sinkhorn_potentials_pnorm(x, y, p, eps, 0.0, its, workspace=ws)
            err[kept].append([float((r.f - f).norm() / f.norm()), float((r.g - g).norm() / g.norm())])
    kept, formed = (np.mean(err[k], axis=0) for k in (True, False))
    assert (kept <= 1.1 * formed).all(), (kept, formed)
