"""Short rounds with many strings, which the blocks share out: string counts around the
line between one block and all, shares of a string or none, strings that become one
phrase in every round, on all SMs and on a few blocks.  Array for array the oracle's."""
import numpy as np
import pytest

import lcg_inputs as li
from oracle import oracle as O

pytestmark = pytest.mark.gpu

ALONE = 2048  # strings that one block takes


def _collection(k, most):
    rng = np.random.default_rng(k)
    lens = rng.integers(2, most + 1, size=k)
    lens[rng.integers(0, k, size=5)] = 3 * most  # a few that go on after the others
    x = li.random_dna(rng, int(lens.sum()))
    return li.from_strings(np.split(x, np.cumsum(lens)[:-1]))


@pytest.mark.parametrize("blocks", [0, 3])
@pytest.mark.parametrize("k,most", [(ALONE - 1, 40), (ALONE, 40), (ALONE + 1, 40), (ALONE + 153, 200), (9_000, 3),
                                    (40_000, 20), (120_000, 6), (30_000, 120)])
def test_many_strings(hf, k, most, blocks):
    from paper_2411_12439_gb300 import Context
    coll = _collection(k, most)
    want = O.build(coll, hf)
    ctx = Context(hf, device=0)
    ctx.selftest_blocks(blocks)
    for _ in range(2):  # round by round, then planned
        g = ctx.build(coll.data, coll.offsets)
        assert O.grammars_equal(g.export(), want.export())
        g.free()
    more = _collection(k // 2, most)
    g = ctx.build(more.data, more.offsets)
    ctx.build_into(g, coll.data, coll.offsets)
    assert O.grammars_equal(g.export(), O.build(more, hf).merge(want).export())
