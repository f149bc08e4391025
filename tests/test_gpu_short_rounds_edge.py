"""Builds whose first round is just inside or just outside the short rounds' range,
and builds whose second or third round is the first inside: array for array the
oracle's, planned or not, and against a resident grammar."""
import numpy as np
import pytest

from test_gpu_short_rounds import _check, _strings

import lcg_inputs as li

pytestmark = pytest.mark.gpu

LAST = 524288  # symbols of the largest round among the short ones


@pytest.mark.parametrize("kind", ["dna", "bytes"])
@pytest.mark.parametrize("n", [LAST - 1, LAST, LAST + 1, 3 * LAST + 7])
def test_edges(hf, n, kind):
    rng = np.random.default_rng(n)
    for k in (1, 9, 40_000):
        _check(hf, li.from_strings(_strings(n, k, kind, rng)), resident=k == 9)


def test_one_run(hf):
    """A string that is one phrase, among the symbols of others."""
    rng = np.random.default_rng(1)
    for n in (LAST - 300_000, LAST):
        s = [np.full(n - 200_000, ord("N"), dtype=np.uint8), li.random_dna(rng, 200_000)]
        _check(hf, li.from_strings(s), resident=True)
