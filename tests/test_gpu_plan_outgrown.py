"""Builds whose planned rounds get fewer places for the next sequence than the strings
need: a context that has seen runs only is given as many bytes of a periodic string,
which has many phrases but few different ones, so no table overflows and it is the
sequence that outgrows its plan.  The build is redone round by round and equals the
oracle's, with the round after it an ordinary or a short one, as launches and as a
graph."""
import numpy as np
import pytest

import lcg_inputs as li
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _runs(n, phrases, k):
    """k strings of n bytes in all with about `phrases` phrases."""
    x = np.full(n, ord("N"), dtype=np.uint8)
    x[:4 * phrases] = np.resize(np.frombuffer(b"ACGT", dtype=np.uint8), 4 * phrases)
    return li.from_strings(np.array_split(x, k))


def _periodic(n, k):
    return li.from_strings(np.array_split(np.resize(np.frombuffer(b"ACGT", dtype=np.uint8), n), k))


# (bytes, phrases of the strings that the plan is made from): the next round is planned
# as a short one of some 4 k, 70 k or 150 k symbols, or as an ordinary one of some 700 k
SIZES = [(530_001, 100), (900_001, 60_000), (1_500_007, 130_000), (6_000_011, 600_000)]


@pytest.mark.parametrize("n,phrases", SIZES)
@pytest.mark.parametrize("k", [1, 7])
@pytest.mark.parametrize("graph", [False, True])
def test_next_sequence_outgrows_its_plan(hf, n, phrases, k, graph):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_12439_gb300 import Context
    few, many = _runs(n, phrases, k), _periodic(n, k)
    want = O.build(many, hf).export()
    ctx = Context(hf, device=0)
    ctx.set_graph(graph)
    buf = torch.from_numpy(few.data.copy()).cuda()
    plan = ctx.build(buf, few.offsets)
    assert not ctx.last_build_stats()["redone"]
    plan.free()
    buf.copy_(torch.from_numpy(many.data))
    torch.cuda.synchronize()
    g = ctx.build(buf, many.offsets)
    st = ctx.last_build_stats()
    assert st["redone"], st
    assert all(r["retries"] == 0 for r in st["per_round"]), st  # no table was too small
    assert O.grammars_equal(g.export(), want)
    g.free()


def test_plan_of_unlike_collections(hf):
    """Rules as long as a string in one collection and hundreds of thousands of short ones
    in the next: a plan made from both asks for no more than a round can have."""
    pytest.importorskip("torch")
    from paper_2411_12439_gb300 import Context
    rng = np.random.default_rng(4)
    runs = _runs(8_000_000, 10, 1)
    noise = li.from_strings([rng.integers(0, 256, size=2_000_000, dtype=np.uint8)])
    last = li.from_strings([li.random_dna(rng, 1_500_000)])
    ctx = Context(hf, device=0)
    for coll in (runs, noise, last, runs, noise):
        g = ctx.build(coll.data, coll.offsets)
        assert O.grammars_equal(g.export(), O.build(coll, hf).export())
        g.free()


@pytest.mark.parametrize("graph", [False, True])
def test_levels_of_short_rounds_outgrow_their_plan(hf, graph):
    """Copies of one string, then as many bytes of unlike ones: the levels of the short
    rounds were planned for a hundredth of the rules."""
    torch = pytest.importorskip("torch")
    from paper_2411_12439_gb300 import Context
    rng = np.random.default_rng(9)
    one = li.random_dna(rng, 4_000)
    copies = li.from_strings([one] * 100)
    unlike = li.from_strings(np.split(li.random_dna(rng, 400_000), 100))
    ctx = Context(hf, device=0)
    ctx.set_graph(graph)
    buf = torch.from_numpy(copies.data.copy()).cuda()
    redone = []
    for coll in (copies, copies, unlike, unlike, copies, unlike):
        buf.copy_(torch.from_numpy(coll.data))
        torch.cuda.synchronize()
        g = ctx.build(buf, coll.offsets)
        redone.append(ctx.last_build_stats()["redone"])
        assert O.grammars_equal(g.export(), O.build(coll, hf).export())
        g.free()
    assert redone == [False, False, True, False, False, False]
