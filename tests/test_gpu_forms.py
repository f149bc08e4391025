"""The packed and the VByte form of grammars whose levels are copied one by one, in
groups, or both: every byte of the packed form from the exported arrays, and grammars
read back from either form equal the one written, and can be merged and built on."""
import numpy as np
import pytest

import lcg_inputs as li
from oracle import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _pad(b):
    return b + bytes(-len(b) % 8)


def _packed(g):
    """The packed form's columns from the exported arrays."""
    out = b""
    for L in g["levels"]:
        out += L["rhs_off"].tobytes() + _pad(L["rhs"].tobytes()) + _pad(L["F"].tobytes())
    return out + _pad(g["c_level"].tobytes()) + _pad(g["c_rank"].tobytes()) + g["F0"].tobytes()


@pytest.mark.parametrize("n,k", [(1, 1), (2, 1), (777, 3), (24_000, 1), (60_001, 20_000), (100_003, 7), (420_000, 2),
                                 (1_200_000, 1)])
@pytest.mark.parametrize("kind", ["dna", "bytes"])
def test_forms(hf, n, k, kind):
    from paper_2411_12439_gb300 import Context
    rng = np.random.default_rng(n)
    cuts = np.linspace(0, n, k + 1).astype(int)
    data = li.random_dna(rng, n) if kind == "dna" else rng.integers(0, 256, size=n, dtype=np.uint8)
    coll = li.from_strings([data[a:b] for a, b in zip(cuts, cuts[1:])])
    ctx = Context(hf, device=0)
    g = ctx.build(coll.data, coll.offsets)
    want = g.export()
    assert O.grammars_equal(want, O.build(coll, hf).export())
    cols = _packed(want)
    plain = np.full(g.packed_size() + 8, 0xAB, dtype=np.uint8)
    pinned = torch.full((g.packed_size() + 8,), 0xAB, dtype=torch.uint8).pin_memory()
    for out in (plain, pinned):
        got = bytes(np.asarray(g.export_packed(out=out)))
        assert got.endswith(cols) and len(got) - len(cols) == 8 * (3 + 2 * len(want["levels"]))
        assert (np.asarray(out)[-8:] == 0xAB).all()
    for h in (ctx.import_vbyte(g.export_vbyte()), ctx.import_vbyte(g.export_vbyte(device=True)),
              ctx.import_packed(np.asarray(g.export_packed()))):
        assert O.grammars_equal(h.export(), want)
        ctx.merge(h, g)
        ctx.build_into(h, coll.data, coll.offsets)
        assert h.export()["c_rank"].size == 3 * k
        assert all(np.array_equal(x["rhs"], y["rhs"]) for x, y in zip(h.export()["levels"], want["levels"]))
        h.free()
    g.free()
    ctx.close()
