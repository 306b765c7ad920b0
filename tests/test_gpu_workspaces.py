"""A workspace of a mixed precision serves the float32 calls: the caller's buffer is used, with the
results of the full one. Tolerance: as in test_gpu_grid.py, 2^-21 (4 max |x~|^2 / eps + 16) relative
for a sum (both sides), times the targets' spread for a map."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_05061_gb300 import native as nat  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


@pytest.mark.parametrize("n,m,d", [(3500, 3300, 16), (2500, 2700, 64), (1700, 1900, 200), (1100, 900, 300), (9000, 3000, 2)])
def test_float32_calls_in_a_mixed_workspace(n, m, d, monkeypatch):
    rng = np.random.default_rng(d)
    x, y = dev(rng.standard_normal((n, d))), dev(rng.standard_normal((m, d)))
    eps = 0.2 * d
    f, g = torch.zeros(n, device="cuda"), dev(rng.standard_normal(m) * eps)
    r2 = float(max((x * x).sum(1).max(), (y * y).sum(1).max()))
    tol = 2 * 2.0 ** -21 * (4 * 1.2 * r2 / eps + 16)

    def calls(ws):
        row, col, _ = nat.coupling_marginals(x, y, f, g, eps, workspace=ws)
        met = nat.coupling_metrics(x, y, f, g, eps, workspace=ws)
        out = nat.entropic_map_apply(x, y, torch.stack([g] * 3), [eps] * 3, [1 / 3, 1 / 2, 1.0], workspace=ws)
        sol = nat.progot_solve(x, y, [0.5, 1.0], [2 * eps, eps], [0.0, 0.0], 4, workspace=ws)
        pn = nat.sinkhorn_potentials_pnorm(x, y, 1.5, eps, 0.0, 3, workspace=ws)
        return row, col, met, out, sol, pn

    full = calls(nat.Workspace(n, m, d))
    ws = nat.Workspace(n, m, d, "bf16x3")
    assert ws.bytes < nat.workspace_size(n, m, d)

    def refuse(*args, **kw):
        raise AssertionError("a workspace of its own")

    monkeypatch.setattr(nat, "Workspace", refuse)
    row, col, met, out, sol, pn = calls(ws)
    torch.testing.assert_close(row, full[0], rtol=tol, atol=0)
    torch.testing.assert_close(col, full[1], rtol=tol, atol=0)
    assert abs(met["mass"] - full[2]["mass"]) <= tol * full[2]["mass"]
    torch.testing.assert_close(out, full[3], rtol=0, atol=3 * tol * r2 ** 0.5)
    torch.testing.assert_close(sol.x_out, full[4].x_out, rtol=0, atol=2 * 2 * 4 * tol * r2 ** 0.5)
    torch.testing.assert_close(pn.f, full[5].f, rtol=0, atol=6 * eps * tol)


def test_marginals_in_the_least_workspace():
    """CUDA cores, without the grid's operands."""
    n, m, d = 1300, 1100, 16
    rng = np.random.default_rng(1)
    x, y = dev(rng.standard_normal((n, d))), dev(rng.standard_normal((m, d)))
    eps = 0.2 * d
    f, g = torch.zeros(n, device="cuda"), dev(rng.standard_normal(m) * eps)
    ws = nat.Workspace(n, m, d)
    full = nat.coupling_marginals(x, y, f, g, eps, workspace=ws)
    ws.bytes = int(nat.lib().progot_workspace_size_min(n, m, d, 0))
    least = nat.coupling_marginals(x, y, f, g, eps, workspace=ws)
    r2 = float(max((x * x).sum(1).max(), (y * y).sum(1).max()))
    tol = 2 * 2.0 ** -21 * (4 * 1.2 * r2 / eps + 16)
    for a, b in zip(least[:2], full[:2]):
        torch.testing.assert_close(a, b, rtol=tol, atol=0)


def test_private_workspace_belongs_to_the_calls_stream(monkeypatch):
    """Dropped when the call returns, it must not go to work on another stream."""
    seen = []
    empty = torch.empty

    def record(*args, **kw):
        if kw.get("dtype") is torch.uint8:
            seen.append(torch.cuda.current_stream().cuda_stream)
        return empty(*args, **kw)

    monkeypatch.setattr(torch, "empty", record)
    x = torch.randn(500, 8, device="cuda")
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    nat.entropic_map_apply(x, x, torch.zeros(1, 500, device="cuda"), [1.0], [1.0], stream=s)
    nat.sinkhorn_potentials(x, x, 1.0, 0.0, 2, stream=s)
    torch.cuda.synchronize()
    assert seen == [s.cuda_stream] * 2


def schedule(x, y, K=2):
    c = float((x ** 2).sum(1).mean() + (y ** 2).sum(1).mean())
    return [1.0 / (K - k) for k in range(K)], [0.2 * c * (K - k) for k in range(K)]


def test_a_server_reserves_for_wide_float32_solves_what_they_use():
    """They run on CUDA cores: two requests fit where their tensor-core parts would leave one."""
    n, d = 2048, 200
    rng = np.random.default_rng(0)
    x, y = rng.standard_normal((n, d)).astype(np.float32), rng.standard_normal((n, d)).astype(np.float32)
    al, eps = schedule(x, y)
    io = 4 * (3 * n * d + 2 * n + n) + 8 * 256
    least = int(nat.lib().progot_workspace_size_min(n, n, d, 0)) + 256
    budget = 2 * (least + io)
    assert budget < 2 * nat.workspace_size(n, n, d)
    srv = nat.Server(budget, n_workers=2, precision="fp32", max_iter=30)
    try:
        ids = [srv.submit(x, y, al, eps, [0.0] * 2) for _ in range(4)]
        outs = [srv.wait(i) for i in ids]
        assert srv.stats()["peak_bytes"] > least + io  # two at a time
    finally:
        srv.close()
    solo = nat.progot_solve(dev(x), dev(y), al, eps, [0.0] * 2, max_iter=30)
    for o in outs:
        np.testing.assert_array_equal(o["x_out"], solo.x_out.cpu().numpy())


@pytest.mark.parametrize("d", [16, 200])
def test_batched_float32_solves_in_the_least_workspace(d):
    rng = np.random.default_rng(d)
    probs = []
    for n, m in ((700, 600), (300, 900), (1100, 130)):
        x, y = rng.standard_normal((n, d)).astype(np.float32), rng.standard_normal((m, d)).astype(np.float32)
        al, eps = schedule(x, y)
        probs.append(dict(x=dev(x), y=dev(y), alpha=al, eps=eps, tau=[0.0] * 2))
    full = nat.progot_solve_batched(probs, max_iter=5, precision="fp32", n_streams=2)
    arr, outs = nat._batch_structs(probs)
    least = max(int(nat.lib().progot_workspace_size_min(p["x"].shape[0], p["y"].shape[0], d, 0)) for p in probs)
    size = 2 * ((least + 255) // 256 * 256)
    for give, status in ((size, nat.PROGOT_ERR_NOT_CONVERGED), (size - 256, nat.PROGOT_ERR_WORKSPACE)):
        buf = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
        base = (buf.data_ptr() + 255) // 256 * 256
        rc = nat.lib().progot_solve_batched(arr, len(probs), 5, 0, 2, base, give, None)
        torch.cuda.synchronize()
        assert rc == status
    for a, b, p in zip(nat._batch_results(arr, outs), full, probs):
        r2 = float(max((p["x"] ** 2).sum(1).max(), (p["y"] ** 2).sum(1).max()))
        tol = 2 * 2 * 5 * 2.0 ** -21 * (4 * 1.2 * r2 / p["eps"][-1] + 16)
        torch.testing.assert_close(a["x_out"], b["x_out"], rtol=0, atol=tol * r2 ** 0.5)
