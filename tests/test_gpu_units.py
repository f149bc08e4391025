"""The parse's units (an eighth of a parse tile per warp) and the ids between
the rounds, at their edges: strings that start, end or retire at and around a
unit's first and last position, more phrases than a warp's queue takes at
once, phrases that reach past the staged symbols, first occurrences that
another warp sees later, and builds against a resident grammar (ids of
resident rules and of new ones in one sequence).  Every grammar equals the
oracle's, array for array."""
import numpy as np
import pytest

import lcg_inputs as li
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _edges(u, rng):
    lens = [u, u - 1, u + 1, 2 * u, 8 * u, 8 * u - 1, 8 * u + 1, 3, 2, u // 2, 17 * u + 5]
    return [li.random_dna(rng, n) for n in lens]


def _retiring(u, rng):
    # short strings, so that some retire in every round, between longer ones
    return [li.random_dna(rng, int(n)) for n in rng.integers(2, 2 * u, size=400)]


def _runs(u, rng):
    # phrases that end in, at and past the staged halo, and equal ones far apart
    out = [np.frombuffer(b"N" * n, dtype=np.uint8) for n in (31, 32, 33, 63, 64, 65)]
    parts = []
    for n in (31, 32, 33, 62, 63, 64, 65, 66, u - 1, u, 5 * u):
        parts += [li.random_dna(rng, u - 7), np.full(n, ord("N"), dtype=np.uint8)]
    return out + [np.concatenate(parts + parts)]


def _text(u, rng):
    # most phrases are new or miss the block's cache: the queue fills again and again
    t = li.zipf_text(rng, 60 * u, copy_frac=0.0)
    return [t, t[::-1].copy(), li.zipf_text(rng, 40 * u)]


@pytest.mark.parametrize("make", [_edges, _retiring, _runs, _text])
@pytest.mark.parametrize("tile", [1024, 2048, 4096])
def test_units(hf, tile, make):
    from paper_2411_12439_gb300 import Context
    rng = np.random.default_rng(tile)
    coll = li.from_strings(make(tile // 8, rng))
    want = O.build(coll, hf).export()
    ctx = Context(hf, device=0)
    ctx.set_tuning(parse_tile=tile, parse_tile_min=0)
    for _ in range(2):  # round by round, then planned
        g = ctx.build(coll.data, coll.offsets)
        assert O.grammars_equal(g.export(), want)
        g.free()
    # halves into one resident grammar
    cut = coll.k // 2
    a, b = coll.subset(range(cut)), coll.subset(range(cut, coll.k))
    g = ctx.build(a.data, a.offsets)
    ctx.build_into(g, b.data, b.offsets)
    assert O.grammars_equal(g.export(), want)
