"""Expansions whose levels pass through the sizes where a block, one launch and a
launch per level take over from one another, with rules too long for a thread in
each: the strings come back, into device and host buffers, exact or too small."""
import numpy as np
import pytest

import lcg_inputs as li

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _strings(rng, n):
    """DNA, DNA with runs of every length, and bytes, of about n each."""
    runs = []
    while sum(x.size for x in runs) < n:
        runs.append(li.random_dna(rng, int(rng.integers(1, 200))))
        runs.append(np.full(int(2 ** rng.uniform(0, 15)), ord("N"), dtype=np.uint8))
    return [li.random_dna(rng, n), np.concatenate(runs)[:n], rng.integers(0, 256, size=n, dtype=np.uint8),
            np.full(n, ord("N"), dtype=np.uint8)]


@pytest.mark.parametrize("n", [9_000, 25_000, 200_000, 1_000_000, 3_200_000, 10_000_000, 33_000_000])
def test_strings_come_back(hf, n):
    from paper_2411_12439_gb300 import Context, LCGError
    rng = np.random.default_rng(n)
    coll = li.from_strings(_strings(rng, n))
    ctx = Context(hf, device=0)
    g = ctx.build(coll.data, coll.offsets)
    for j in range(coll.k):
        want = coll.string(j)
        out = torch.full((n + 16,), 0xAB, dtype=torch.uint8, device="cuda")
        assert g.decompress(j, out) == n
        got = out.cpu().numpy()
        assert np.array_equal(got[:n], want) and (got[n:] == 0xAB).all()
        assert g.decompress(j) == want.tobytes()
        try:
            g.decompress(j, torch.empty(n - 1, dtype=torch.uint8, device="cuda"))
            raise AssertionError("a buffer too small was taken")
        except LCGError as e:
            assert e.code == -1
    g.free()
    ctx.close()
