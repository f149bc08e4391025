"""Run-length rules and simplification of grammars whose rules are long (taken by
whole warps past 64 symbols): runs that start, end and meet at the edges of a
warp's 32-symbol words and 256-symbol steps, against the oracle, array for array."""
import numpy as np
import pytest

import lcg_inputs as li
from oracle import oracle as O
from oracle import postprocess as P

pytestmark = pytest.mark.gpu


def _lengths(lens):
    """Runs of the given lengths one after another, two symbols in turn: with a
    family whose fingerprints all collide a string is one rule."""
    return np.concatenate([np.full(n, 65 + (i & 1), dtype=np.uint8) for i, n in enumerate(lens)])


@pytest.mark.parametrize("shift", [0, 1, 31, 32, 33, 255, 256, 257])
def test_long_rules(shift):
    from paper_2411_12439_gb300 import Context
    rng = np.random.default_rng(shift)
    strings = [_lengths([shift + 1, 64, 1, 1, 2, 31, 32, 33, 1, 255, 256, 257, 1]),
               _lengths([shift + 1] + rng.integers(1, 4, size=400).tolist()),
               _lengths([65 + shift]), _lengths([shift + 1, 64]), _lengths([63, 1, shift + 1]),
               _lengths([5000, shift + 1, 5000])]
    for m_bits in (1, 2, 32):
        hf = li.hash_family(m_bits=m_bits)
        coll = li.from_strings(strings)
        ctx = Context(hf, device=0)
        g = ctx.build(coll.data, coll.offsets)
        want = P.postprocess(O.build(coll, hf).export())
        pp = ctx.postprocess(g)
        got = pp.export()
        for key in ("kind", "rhs_off", "rhs", "c"):
            assert np.array_equal(np.asarray(got[key]), np.asarray(want[key])), (m_bits, key)
