"""lcg_decompress at its edges: strings around the sizes that one block expands,
rules too long for one thread, outputs at every alignment within 16 bytes with
their neighbours left alone, host and device buffers, and buffers too small."""
import numpy as np
import pytest

import lcg_inputs as li

pytestmark = pytest.mark.gpu

GUARD = 0xA5


def _cases():
    rng = np.random.default_rng(19)
    dna = lambda n: li.random_dna(rng, n)
    run = lambda n, c=b"N": np.frombuffer(c * n, dtype=np.uint8)
    yield [dna(n) for n in (1, 2, 3, 15, 16, 17, 8191, 8192, 8193, 28_000, 65_535, 65_536, 65_537, 300_001)]
    # rules of 33 symbols and more, in one block, in a tile that is staged, and in one that is not
    yield [run(33), run(65_536), run(65_537), run(400_000),
           np.concatenate([np.concatenate([run(40 + i % 7), dna(9)]) for i in range(1500)]),
           np.concatenate([np.concatenate([run(3000 + i), dna(5), run(33, b"T")]) for i in range(200)])]
    yield [li.zipf_text(rng, n) for n in (100, 9000, 70_001, 200_003)]


@pytest.mark.parametrize("case", range(3))
def test_expand_edges(hf, case):
    import torch
    from paper_2411_12439_gb300 import Context, LCGError
    coll = li.from_strings(list(_cases())[case])
    ctx = Context(hf, device=0)
    g = ctx.build(coll.data, coll.offsets)
    for j in range(coll.k):
        want = coll.string(j)
        n = want.shape[0]
        assert g.decompress(j) == want.tobytes()
        for skew in (0, 1, 7, 15) if n > 20_000 else range(16):
            buf = torch.full((n + 64,), GUARD, dtype=torch.uint8, device="cuda")
            assert g.decompress(j, out=buf[16 + skew:16 + skew + n]) == n
            got = buf.cpu().numpy()
            assert np.array_equal(got[16 + skew:16 + skew + n], want)
            assert np.all(got[:16 + skew] == GUARD) and np.all(got[16 + skew + n:] == GUARD)
        buf = torch.full((n + 16,), GUARD, dtype=torch.uint8, device="cuda")
        with pytest.raises(LCGError) as e:
            g.decompress(j, out=buf[:n - 1])
        assert e.value.code == -1
        assert bool((buf == GUARD).all())  # nothing is written
