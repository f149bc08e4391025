"""A merge that runs out of device memory, at each of its allocations in turn, leaves
G_a as it was: its arrays, its packed and VByte forms, its strings.  The same merge
afterwards equals the oracle's.  The allocation is refused on the host."""
import gc

import numpy as np
import pytest

from test_zz_no_alloc import _cudart, _pool_used

import lcg_inputs as li
from oracle import oracle as O

pytestmark = pytest.mark.gpu

LCG_ENOMEM = -2


def _parts(kind):
    rng = np.random.default_rng(3)
    if kind == "more levels":  # G_b has levels that G_a has not; all of them small
        return [li.random_dna(rng, 40)], [li.random_dna(rng, 60_000), li.random_dna(rng, 500)]
    if kind == "fewer levels":
        return [li.random_dna(rng, 60_000), b"A"], [li.random_dna(rng, 700)]
    # large levels below small ones
    return [rng.integers(0, 256, size=40_000, dtype=np.uint8)], [rng.integers(0, 256, size=1_600_000, dtype=np.uint8)]


@pytest.mark.parametrize("kind", ["more levels", "fewer levels", "large levels"])
def test_every_allocation_of_a_merge(hf, kind):
    from paper_2411_12439_gb300 import Context, LCGError
    ca, cb = (li.from_strings(p) for p in _parts(kind))
    ctx = Context(hf, device=0)
    g = ctx.build(ca.data, ca.offsets)
    before, packed = g.export(), g.export_packed()
    g.free()
    h = ctx.build(cb.data, cb.offsets)
    want = O.build(ca, hf).merge(O.build(cb, hf)).export()
    g = ctx.import_packed(packed)  # (what the context keeps between calls)
    ctx.merge(g, h)
    back = ctx.import_vbyte(g.export_vbyte())
    assert O.grammars_equal(back.export(), want)
    back.free()
    g.free()
    gc.collect()  # (contexts of earlier tests go now, not between two reads of the pool)
    rt = _cudart()
    used = _pool_used(rt)
    refused = 0
    for nth in range(1, 200):
        g = ctx.import_packed(packed)
        ctx.selftest_alloc_failure(nth)
        try:
            ctx.merge(g, h)
            done = True
        except LCGError as e:
            assert e.code == LCG_ENOMEM, e
            done = False
        ctx.selftest_alloc_failure(0)
        if not done:
            refused += 1
            assert O.grammars_equal(g.export(), before)
            assert np.array_equal(np.asarray(g.export_packed()), np.asarray(packed))
            assert O.grammars_equal(ctx.import_vbyte(g.export_vbyte()).export(), before)
            assert g.decompress(0) == ca.string(0).tobytes()
            ctx.merge(g, h)  # the next try succeeds
        assert O.grammars_equal(g.export(), want)
        g.free()
        assert _pool_used(rt) == used  # nothing is left behind
        if done:
            break
    assert done and refused >= 4, refused


def test_packed_form_without_device_memory(hf):
    """The packed form needs no scratch: with none to be had it is copied column by column."""
    from paper_2411_12439_gb300 import Context
    coll = li.from_strings([li.random_dna(np.random.default_rng(1), 20_000)])
    ctx = Context(hf, device=0)
    g = ctx.build(coll.data, coll.offsets)
    want = np.asarray(g.export_packed())
    ctx.selftest_alloc_failure(1)
    assert np.array_equal(np.asarray(g.export_packed()), want)
    ctx.selftest_alloc_failure(0)
