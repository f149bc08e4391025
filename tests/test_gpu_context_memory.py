"""What a context keeps between calls: words of the single-pass scans and of the breaks'
look-ahead, a thousandth of the largest input, and nothing of a build's own."""
import numpy as np
import pytest

from test_zz_no_alloc import _cudart, _pool_used

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True])
def test_kept_after_a_build(hf, graph):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_12439_gb300 import Context
    n = 64_000_000
    g = torch.Generator(device="cuda").manual_seed(2)
    data = torch.randint(0, 4, (n,), dtype=torch.uint8, device="cuda", generator=g)
    off = np.array([0, n // 3, n], dtype=np.uint64)
    rt = _cudart()
    ctx = Context(hf, device=0)
    before = _pool_used(rt)
    ctx.set_graph(graph)
    for _ in range(3):  # round by round, then planned
        ctx.build(data, off).free()
    ctx.set_graph(False)
    assert _pool_used(rt) - before <= n // 500
