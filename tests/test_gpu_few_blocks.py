"""The launches whose blocks wait for one another, with fewer blocks than the work has
steps (a device or a partition with few SMs): short rounds of up to 64 steps of breaks,
with runs that cross them, the small levels of a merge and the middle levels of an
expansion give what the oracle gives."""
import numpy as np
import pytest

import lcg_inputs as li
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _collection(n, k):
    rng = np.random.default_rng(n + k)
    x = li.random_dna(rng, n)
    for at, size in ((n // 9, n // 5), (n // 2, 3), (n // 2 + 100, n // 4)):  # runs over several steps
        x[at:at + size] = ord("N")
    return li.from_strings(np.array_split(x, k))


@pytest.mark.parametrize("most", [1, 2, 5, 63])
@pytest.mark.parametrize("n,k", [(524_288, 1), (524_288, 300), (300_001, 9), (700_001, 4)])
def test_few_blocks(hf, most, n, k):
    from paper_2411_12439_gb300 import Context
    coll, more = _collection(n, k), _collection(n // 3, 2)
    one, two = O.build(coll, hf), O.build(more, hf)
    want = one.export()
    ctx = Context(hf, device=0)
    ctx.selftest_blocks(most)
    for _ in range(2):  # round by round, then planned
        g = ctx.build(coll.data, coll.offsets)
        assert O.grammars_equal(g.export(), want)
    h = ctx.build(more.data, more.offsets)
    merged = one.merge(two).export()
    into = ctx.import_vbyte(g.export_vbyte())
    ctx.build_into(into, more.data, more.offsets)
    assert O.grammars_equal(into.export(), merged)
    ctx.merge(g, h)
    assert O.grammars_equal(g.export(), merged)
    for j in (0, k - 1, k):
        want_s = coll.string(j) if j < k else more.string(0)
        assert g.decompress(j) == want_s.tobytes()
