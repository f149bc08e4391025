"""The short rounds of a build (one launch for all their parses, one for all
their namings; the last of them in one block's shared memory) at the sizes
where they begin, with few and many strings, runs, equal strings and colliding
fingerprints: fresh builds and builds against a resident grammar equal the
oracle's, array for array."""
import numpy as np
import pytest

import lcg_inputs as li
from oracle import oracle as O

pytestmark = pytest.mark.gpu

SOLO, TAIL = 1024, 131072  # symbols


def _strings(n, k, kind, rng):
    """k strings of n bytes in all (two or more each)."""
    cuts = np.sort(rng.choice(np.arange(1, n // 2), size=k - 1, replace=False)) * 2 if k > 1 else np.zeros(0, int)
    lens = np.diff(np.concatenate([[0], cuts, [n]]))
    if kind == "dna":
        return [li.random_dna(rng, int(m)) for m in lens]
    if kind == "runs":  # equal strings, and phrases as long as a string
        return [np.full(int(m), ord("N"), dtype=np.uint8) for m in lens]
    return [rng.integers(0, 256, size=int(m), dtype=np.uint8) for m in lens]


def _check(hf, coll, resident):
    from paper_2411_12439_gb300 import Context
    want = O.build(coll, hf).export()
    ctx = Context(hf, device=0)
    for _ in range(2):  # round by round, then planned
        g = ctx.build(coll.data, coll.offsets)
        assert O.grammars_equal(g.export(), want)
        g.free()
    if resident and coll.k > 1:
        cut = coll.k // 2
        a, b = coll.subset(range(cut)), coll.subset(range(cut, coll.k))
        g = ctx.build(a.data, a.offsets)
        for _ in range(2):  # the second time every phrase is resident
            ctx.build_into(g, b.data, b.offsets)
        ab = li.from_strings([a.string(j) for j in range(a.k)] + 2 * [b.string(j) for j in range(b.k)])
        assert O.grammars_equal(g.export(), O.build(ab, hf).export())


@pytest.mark.parametrize("kind", ["dna", "runs", "bytes"])
@pytest.mark.parametrize("n", [2, 3, 31, 33, SOLO - 1, SOLO, SOLO + 1, 3 * SOLO, 8192, 8193, 20_011])
def test_small_builds(hf, n, kind):
    rng = np.random.default_rng(n)
    for k in sorted({1, 2, min(7, n // 2), n // 3, n // 2}):
        if 1 <= k <= n // 2:
            _check(hf, li.from_strings(_strings(n, k, kind, rng)), resident=True)


@pytest.mark.parametrize("n", [TAIL - 1, TAIL, TAIL + 1, 3 * TAIL])
def test_first_short_round(hf, n):
    rng = np.random.default_rng(n)
    for k in (1, 5, 3000):
        _check(hf, li.from_strings(_strings(n, k, "dna", rng)), resident=k == 5)


@pytest.mark.parametrize("m_bits", [1, 2, 5])
def test_colliding_fingerprints(m_bits):
    hf = li.hash_family(m_bits=m_bits)
    rng = np.random.default_rng(m_bits)
    for n, k in ((500, 3), (900, 200), (5000, 11)):
        _check(hf, li.from_strings(_strings(n, k, "bytes", rng)), resident=True)
