"""What a context keeps between calls: words of the single-pass scans and of the breaks'
look-ahead, a thousandth of the largest input, and nothing of a build's own."""
import gc

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
    gc.collect()  # (contexts of earlier tests go now, not between two reads of the pool)
    rt = _cudart()
    ctx = Context(hf, device=0)
    before = _pool_used(rt)
    ctx.set_graph(graph)
    for _ in range(3):  # round by round, then planned
        ctx.build(data, off).free()
    ctx.set_graph(False)
    assert _pool_used(rt) - before <= n // 500


@pytest.mark.parametrize("kind", ["copies", "dna", "bytes", "short"])
def test_kept_by_a_grammar(hf, kind):
    """A grammar's memory is what its arrays need, a few times over, not what the rounds of
    its build could have needed."""
    pytest.importorskip("torch")
    import lcg_inputs as li
    from paper_2411_12439_gb300 import Context
    rng = np.random.default_rng(6)
    one = li.random_dna(rng, 5_000)
    coll = li.from_strings({"copies": [one] * 100, "dna": [li.random_dna(rng, 500_000)],
                            "bytes": [rng.integers(0, 256, size=400_000, dtype=np.uint8)], "short": [one[:300]]}[kind])
    gc.collect()  # (contexts of earlier tests go now, not between two reads of the pool)
    rt = _cudart()
    ctx = Context(hf, device=0)
    for graph in (None, False, True):  # round by round, planned, a graph's
        ctx.set_graph(bool(graph))
        if graph is not None:
            ctx.build(coll.data, coll.offsets).free()
        before = _pool_used(rt)
        g = ctx.build(coll.data, coll.offsets)
        held = _pool_used(rt) - before
        assert held <= 4 * g.packed_size() + 600_000, (graph, held, g.packed_size())
        g.free()


def test_replaced_graph_keeps_its_grammar_only(hf):
    """A graph that goes while the grammar of its last launch is in use gives the memory
    of its rounds back at once, and the rest with the grammar."""
    torch = pytest.importorskip("torch")
    from paper_2411_12439_gb300 import Context
    import ctypes
    gc.collect()  # (contexts of earlier tests go now, not between two reads of the pool)
    rt = _cudart()

    def reserved():  # by graphs, on the device
        torch.cuda.synchronize()
        x = ctypes.c_uint64()
        attr_reserved_mem_current = 2  # cudaGraphMemAttrReservedMemCurrent
        assert rt.cudaDeviceGetGraphMemAttribute(0, attr_reserved_mem_current, ctypes.byref(x)) == 0
        return x.value

    n = 64_000_000
    g = torch.Generator(device="cuda").manual_seed(2)
    data = torch.randint(0, 4, (n,), dtype=torch.uint8, device="cuda", generator=g)
    off = np.array([0, n // 3, n], dtype=np.uint64)
    torch.cuda.synchronize()
    ctx = Context(hf, device=0)
    ctx.build(data, off).free()
    before = reserved()
    ctx.set_graph(True)
    grammar = ctx.build(data, off)
    assert ctx.last_build_stats()["graph"] == 1
    want = grammar.export_packed()
    full = reserved() - before
    ctx.set_graph(False)
    held = reserved() - before
    assert full > 2 * n and held < full // 2, (full, held)
    ctx.build(data, off).free()
    assert np.array_equal(np.asarray(grammar.export_packed()), np.asarray(want))
    grammar.free()
    assert reserved() <= before
