"""Which workspace a float32 call accepts (host arithmetic only)."""
import pytest

from paper_2406_05061_gb300 import native


@pytest.mark.parametrize("n,m", [(1, 1), (127, 129), (500, 20000), (8192, 8192), (65536, 40000)])
@pytest.mark.parametrize("d", [1, 16, 64, 65, 256, 257, 1024, 3072])
def test_a_mixed_workspace_covers_a_float32_call(n, m, d):
    least = native.lib().progot_workspace_size_min(n, m, d, native.PRECISIONS["fp32"])
    mixed = native.workspace_size(n, m, d, "bf16x3")
    assert 0 < least <= min(mixed, native.workspace_size(n, m, d, "fp32"))
    for precision in ("bf16x3", "bf16"):
        assert native.lib().progot_workspace_size_min(n, m, d, native.PRECISIONS[precision]) == native.workspace_size(n, m, d, precision)


@pytest.mark.parametrize("d", [65, 256, 1024])
def test_batched_float32_solves_reserve_what_they_use(d):
    """Beyond d = 64 they run on CUDA cores; every problem's own need counts, not the largest sizes together."""
    import numpy as np

    x, y, K = np.zeros((4000, d), np.float32), np.zeros((300, d), np.float32), 2
    arr = (native.ProblemStruct * 2)()
    for i, (p, q) in enumerate(((x, y), (y, x))):
        arr[i], _ = native._problem_struct(p, q, [0.5, 1.0], [1.0] * K, [0.0] * K, np.empty_like(p),
                                           np.empty((K, len(q)), np.float32))
    need = max(int(native.lib().progot_workspace_size_min(len(p), len(q), d, 0)) for p, q in ((x, y), (y, x)))
    assert native.lib().progot_batched_workspace_size(arr, 2, 0, 3) == 3 * ((need + 255) // 256 * 256) + 256
