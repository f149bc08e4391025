"""Merges at the sizes where a level is handled another way: rules read by a
thread or by a warp, keys that hold their symbols or hash them, levels that fit
their arrays, that grow ahead of what is added and that wait for it, G_b a part
of G_a, equal to it, or empty of new rules.  Array for array the oracle's."""
import numpy as np
import pytest

import lcg_inputs as li
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _runs(rng, lens):
    """Strings with runs of one byte (a rule each, as long as the run) in DNA."""
    out = []
    for m in lens:
        parts = [li.random_dna(rng, int(rng.integers(1, 40))), np.full(m, ord("N"), dtype=np.uint8),
                 li.random_dna(rng, int(rng.integers(1, 40)))]
        out.append(np.concatenate(parts))
    return out


def _check(ctx, hf, *parts, form=None):
    want = O.build(li.from_strings(parts[0]), hf)
    g = ctx.build(li.from_strings(parts[0]).data, li.from_strings(parts[0]).offsets)
    for p in parts[1:]:
        c = li.from_strings(p)
        h = ctx.build(c.data, c.offsets)
        if form == "vbyte":
            h = ctx.import_vbyte(h.export_vbyte())
        ctx.merge(g, h)
        want = want.merge(O.build(c, hf))
        assert O.grammars_equal(g.export(), want.export())
    # the level tables hold the appended rules: a build against them finds them all
    c = li.from_strings(parts[-1])
    ctx.build_into(g, c.data, c.offsets)
    assert O.grammars_equal(g.export(), want.merge(O.build(c, hf)).export())


@pytest.fixture()
def ctx(hf):
    from paper_2411_12439_gb300 import Context
    return Context(hf, device=0)


@pytest.mark.parametrize("form", [None, "vbyte"])
def test_rule_lengths(ctx, hf, form):
    rng = np.random.default_rng(5)
    edges = [1, 2, 4, 5, 13, 14, 15, 31, 32, 33, 63, 64, 65, 127, 129, 1000, 5003]
    a, b = _runs(rng, edges), _runs(rng, edges[1::2] + [40, 41, 7001])
    _check(ctx, hf, a, b, a, form=form)
    _check(ctx, hf, a[:1], a, b, form=form)


@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 2049, 100_000])
def test_sizes(ctx, hf, n):
    rng = np.random.default_rng(n)
    a, b = [li.random_dna(rng, n)], [li.random_dna(rng, n + 1), li.random_dna(rng, max(1, n // 3))]
    _check(ctx, hf, a, b, a, b)
    _check(ctx, hf, b, a)


@pytest.mark.parametrize("n", [2_200_000, 4_000_000])
def test_large_levels(ctx, hf, n):
    """Random bytes: nearly every phrase is a rule of its own, about a third of n."""
    rng = np.random.default_rng(n)
    a, b = (rng.integers(0, 256, size=n, dtype=np.uint8) for _ in range(2))
    _check(ctx, hf, [a], [b, a[: n // 2]], [b])
