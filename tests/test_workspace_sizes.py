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
