"""The VByte kernels at the edges of their tiles (2048 values, 4096 stream bytes,
four of either to a counting block) and of the 16-byte lines of the output, for
streams of shortest, longest and mixed values; values that reach over the edge of a
tile, whole and malformed."""
import gc

import numpy as np
import pytest

import lcg_inputs as li
from oracle import vbyte as V

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2411_12439_gb300 import Context, LCGError  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    yield Context(li.hash_family(), device=0)
    gc.collect()  # tensors held by the tracebacks of refused calls go now, not in a later test


def _values(kind, n):
    rng = np.random.default_rng(n)
    if kind == "short":
        return rng.integers(0, 128, size=n, dtype=np.uint32)
    if kind == "long":
        return rng.integers(1 << 28, 1 << 32, size=n, dtype=np.uint64).astype(np.uint32)
    return (rng.integers(0, 1 << 32, size=n, dtype=np.uint64) >> rng.integers(0, 32, size=n).astype(np.uint64)).astype(
        np.uint32)


def _bytes(b, shift=0):
    t = torch.zeros(len(b) + shift + 16, dtype=torch.uint8, device="cuda")
    t[shift:shift + len(b)] = torch.from_numpy(np.frombuffer(b, dtype=np.uint8).copy()).cuda()
    return t[shift:shift + len(b)]


def _code(ctx, b, n):
    try:
        ctx.vbyte_decode(_bytes(b), n)
    except LCGError as e:
        return e.code
    return 0


@pytest.mark.parametrize("kind", ["short", "long", "mixed"])
@pytest.mark.parametrize("n", [1, 3, 15, 16, 17, 819, 820, 2048, 4095, 4096, 4097, 8191, 8192, 8193, 16383, 16385, 40_000])
def test_sizes(ctx, kind, n):
    v = _values(kind, n)
    want = V.encode_np(v)
    got = ctx.vbyte_encode(torch.from_numpy(v.view(np.int32)).cuda())
    assert got.cpu().numpy().tobytes() == want
    assert np.array_equal(ctx.vbyte_decode(_bytes(want), n).cpu().numpy().view(np.uint32), v)


@pytest.mark.parametrize("kind", ["short", "long", "mixed"])
@pytest.mark.parametrize("shift", range(1, 16))
def test_output_lines(ctx, kind, shift):
    for n in (1, 2, 5, 20, 2049):
        v = _values(kind, n)
        want = V.encode_np(v)
        big = torch.full((len(want) + 64,), 0xAB, dtype=torch.uint8, device="cuda")
        got = ctx.vbyte_encode(torch.from_numpy(v.view(np.int32)).cuda(), out=big[shift:])
        assert got.cpu().numpy().tobytes() == want
        rest = torch.cat([big[:shift], big[shift + len(want):]])
        assert bool((rest == 0xAB).all())
        assert np.array_equal(ctx.vbyte_decode(_bytes(want, shift), n).cpu().numpy().view(np.uint32), v)


@pytest.mark.parametrize("before", range(4088, 4100))
def test_values_over_a_tile_edge(ctx, before):
    lead = bytes(before)  # values of one byte
    for tail in ("ffffffff0f", "8001", "80808001", "8080808001"):
        b = lead + bytes.fromhex(tail) + bytes(3)
        want = np.zeros(before + 4, dtype=np.uint32)
        want[before] = sum((x & 0x7F) << (7 * j) for j, x in enumerate(bytes.fromhex(tail)))
        assert np.array_equal(ctx.vbyte_decode(_bytes(b), before + 4).cpu().numpy().view(np.uint32), want)
    for tail in ("808080808000", "ffffffff10", "ffffffffffffffffffff00", "80" * 20 + "00"):
        assert _code(ctx, lead + bytes.fromhex(tail), before + 1) == -1
    assert _code(ctx, lead + b"\x80", before + 1) == -1
