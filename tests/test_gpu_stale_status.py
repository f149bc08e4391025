"""An error of one call does not carry over into the next: after a rejected VByte stream
(and after a wait that ran out) a good grammar's strings, short and long, come back
through both entry points, and an expansion that is refused leaves no memory behind."""
import gc

import numpy as np
import pytest

from test_zz_no_alloc import _cudart, _pool_used

import lcg_inputs as li

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def built(hf):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_12439_gb300 import Context
    rng = np.random.default_rng(12)
    # one block's, one launch's for the middle levels, and level by level
    coll = li.from_strings([li.random_dna(rng, n) for n in (500, 200_000, 1_000_000, 9_000_000)])
    ctx = Context(hf, device=0)
    return ctx, ctx.build(coll.data, coll.offsets), coll


def _reject_stream(ctx):
    import torch
    from paper_2411_12439_gb300 import LCGError
    bad = torch.full((64,), 0x80, dtype=torch.uint8, device="cuda")  # no value ends
    with pytest.raises(LCGError) as e:
        ctx.vbyte_decode(bad, 20)
    assert e.value.code == -1


@pytest.mark.parametrize("spoil", [_reject_stream, lambda ctx: ctx.selftest_wait_timeout()])
@pytest.mark.parametrize("j", [0, 1, 2, 3])
def test_expansion_after_a_failed_call(built, spoil, j):
    import torch
    ctx, g, coll = built
    want = coll.string(j)
    spoil(ctx)
    assert g.decompress(j) == want.tobytes()
    spoil(ctx)
    out = torch.zeros(want.size, dtype=torch.uint8, device="cuda")
    assert g.decompress(j, out) == want.size
    assert np.array_equal(out.cpu().numpy(), want)
    if want.size <= 1 << 20:
        spoil(ctx)
        out.zero_()
        torch.cuda.synchronize()
        assert g.decompress_static(j, out) == want.size
        assert np.array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("j", [1, 2, 3])
def test_refused_expansion_returns_its_scratch(built, j):
    import torch
    from paper_2411_12439_gb300 import LCGError
    ctx, g, coll = built
    gc.collect()  # (contexts of earlier tests go now, not between two reads of the pool)
    rt = _cudart()
    small = torch.zeros(coll.string(j).size - 1, dtype=torch.uint8, device="cuda")
    used = _pool_used(rt)
    for _ in range(3):
        with pytest.raises(LCGError):
            g.decompress(j, small)
    assert _pool_used(rt) == used


def test_string_of_one_byte_in_a_deep_grammar(hf):
    """More than 64 levels, and a string that is a byte: in its place when the call is
    back, for a reader on another stream."""
    import torch
    from paper_2411_12439_gb300 import Context
    family = li.hash_family(levels=80)
    ctx = Context(family, device=0)

    # level i's only rule is level i - 1's; level 1's is the byte 65
    levels, below = [], None
    for i in range(1, 71):
        below = _fingerprint(family, i, 65 if i == 1 else 0, below)
        levels.append({"g": 1, "rhs_off": np.array([0, 1], dtype=np.uint64),
                       "rhs": np.array([65 if i == 1 else 0], dtype=np.uint32),
                       "F": np.array([below], dtype=np.uint32)})
    g = ctx.import_grammar({"levels": levels, "c_level": np.array([0, 70], dtype=np.uint32),
                            "c_rank": np.array([66, 0], dtype=np.uint32)})
    other = torch.cuda.Stream()
    for j, byte in ((0, 66), (1, 65)):
        assert g.decompress(j) == bytes([byte])
        for _ in range(50):
            out = torch.zeros(1, dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            assert g.decompress(j, out) == 1
            with torch.cuda.stream(other):
                assert int(out.item()) == byte


def _fingerprint(family, i, symbol, below):
    """h^i of a rule of one symbol (Eq. fast_hash over the level below)."""
    p = (1 << 61) - 1
    a, b = int(family.a[i]), int(family.b[i])
    if i == 1:
        below = (int(family.a[0]) * symbol + int(family.b[0])) % p % (1 << int(family.m_bits))
    return (a * int(below) + b) % p % (1 << int(family.m_bits))
