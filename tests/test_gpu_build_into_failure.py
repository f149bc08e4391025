"""A parse against a resident grammar that fails, for lack of memory at any of its
allocations or of hash functions, leaves the grammar as it was, and the next one extends
it as if nothing had been."""
import gc

import numpy as np
import pytest

from test_zz_no_alloc import _cudart, _pool_used

import lcg_inputs as li
from oracle import oracle as O

pytestmark = pytest.mark.gpu

LCG_ENOMEM, LCG_ELEVELS = -2, -3


def _collections(n):
    rng = np.random.default_rng(n)
    a = li.from_strings([li.random_dna(rng, 3000), b"C"])
    b = li.from_strings([li.random_dna(rng, n), a.string(0), b"G", li.random_dna(rng, 50)])
    both = li.from_strings([c.string(j) for c in (a, b) for j in range(c.k)])
    return a, b, both


@pytest.mark.parametrize("n", [40_000, 700_000])  # short rounds only; ordinary ones first
def test_every_allocation_of_a_parse(hf, n):
    from paper_2411_12439_gb300 import Context, LCGError
    a, b, both = _collections(n)
    ctx = Context(hf, device=0)
    g = ctx.build(a.data, a.offsets)
    before = g.export()
    want = O.build(both, hf).export()
    refused = 0
    for nth in range(1, 300):
        ctx.selftest_alloc_failure(nth)
        try:
            ctx.build_into(g, b.data, b.offsets)
            break
        except LCGError as e:
            assert e.code == LCG_ENOMEM, e
        finally:
            ctx.selftest_alloc_failure(0)
        refused += 1
        assert O.grammars_equal(g.export(), before)
    assert refused >= 4
    assert O.grammars_equal(g.export(), want)


def test_too_few_hash_functions():
    from paper_2411_12439_gb300 import Context, LCGError
    hf = li.hash_family(levels=5)
    ctx = Context(hf, device=0)
    a = li.from_strings([b"ACGTACGGT", b"T"])
    long = li.from_strings([li.random_dna(np.random.default_rng(2), 90_000), b"ACG"])
    g = ctx.build(a.data, a.offsets)
    before = g.export()
    for _ in range(2):
        with pytest.raises(LCGError) as e:
            ctx.build_into(g, long.data, long.offsets)
        assert e.value.code == LCG_ELEVELS
        assert O.grammars_equal(g.export(), before)
    ctx.build_into(g, a.data, a.offsets)
    both = li.from_strings(2 * [a.string(j) for j in range(a.k)])
    assert O.grammars_equal(g.export(), O.build(both, hf).export())


@pytest.mark.parametrize("n", [40_000, 700_000, 3_000_000])
@pytest.mark.parametrize("mode", ["first", "planned", "graph", "resident"])
def test_failed_builds_keep_no_memory(hf, n, mode):
    """Every allocation of a build refused in turn: what the build had is given back."""
    from paper_2411_12439_gb300 import Context, LCGError
    a, b, _ = _collections(n)
    gc.collect()  # (contexts of earlier tests go now, not between two reads of the pool)
    rt = _cudart()
    ctx = Context(hf, device=0)
    g = ctx.build(a.data, a.offsets)
    want = O.build(b, hf).export()
    if mode in ("planned", "graph"):
        ctx.build(b.data, b.offsets).free()
    ctx.build_into(g, b.data, b.offsets)  # (what the context and the grammar keep)
    before = g.export()
    refused = 0
    for nth in range(1, 400):
        c = Context(hf, device=0) if mode == "first" else ctx
        c.set_graph(mode == "graph")
        used = []
        # at first arrays of the resident grammar, the words of the scans (one more of
        # them each time) or the upload buffer may grow, which are kept
        for _ in range(6):
            c.selftest_alloc_failure(nth)
            try:
                if mode == "resident":
                    c.build_into(g, b.data, b.offsets)
                else:
                    h = c.build(b.data, b.offsets)
                    assert O.grammars_equal(h.export(), want)
                    h.free()
                break
            except LCGError as e:
                assert e.code == LCG_ENOMEM, e
            finally:
                c.selftest_alloc_failure(0)
            used.append(_pool_used(rt))
            if mode == "resident":
                assert O.grammars_equal(g.export(), before)
        c.set_graph(False)
        if len(used) < 6:
            break
        refused += 1
        assert used[-1] == used[-2], (nth, used)
    assert len(used) < 6 and refused >= 4
