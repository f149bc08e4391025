"""Families with so few fingerprint bits that long phrases share their hashes by the
thousand: chains of equal keys in tables that are far from full, in ordinary and short
rounds, built without hints, from a plan, and from hints of larger alphabets.  Array for
array the oracle's."""
import numpy as np
import pytest

import lcg_inputs as li
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _collection(kind, n, k):
    rng = np.random.default_rng(n)
    if kind == "dna":
        x = li.random_dna(rng, n)
    elif kind == "bytes":
        x = rng.integers(0, 256, size=n, dtype=np.uint8)
    else:
        x = li.zipf_text(rng, n)
    return li.from_strings(np.array_split(x, k))


@pytest.mark.parametrize("m_bits", [1, 2])
@pytest.mark.parametrize("kind", ["dna", "bytes", "text"])
@pytest.mark.parametrize("n,k", [(500_000, 1), (1_900_000, 1), (2_480_000, 16)])
def test_shared_hashes(m_bits, kind, n, k):
    from paper_2411_12439_gb300 import Context
    hf = li.hash_family(m_bits=m_bits)
    coll = _collection(kind, n, k)
    want = O.build(coll, hf).export()
    ctx = Context(hf, device=0)
    for _ in range(2):  # round by round, then planned
        g = ctx.build(coll.data, coll.offsets)
        assert O.grammars_equal(g.export(), want)
        g.free()
