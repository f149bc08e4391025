"""Grammars of captured graphs, kept while their context captures other graphs, turns
graphs off or is closed, beside other contexts that do the same: none is changed by what
the others build, and all read back as the oracle's."""
import random

import numpy as np
import pytest

import lcg_inputs as li
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _collections(hf):
    rng = np.random.default_rng(21)
    out = []
    for n, k in ((4, 2), (9_000, 490), (60_000, 3), (540_000, 63), (1_600_000, 4)):
        c = li.from_strings(np.array_split(li.random_dna(rng, n), k))
        out.append((c, O.build(c, hf).export()))
    return out


def test_a_graph_outlives_its_grammar(hf):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_12439_gb300 import Context
    colls = _collections(hf)
    r = random.Random(3)
    ctxs, kept, launches = [], [], 0
    for step in range(400):
        if len(ctxs) < 3:
            ctxs.append(Context(hf, device=0))
            ctxs[-1].set_graph(True)
        ctx = r.choice(ctxs)
        c, want = r.choice(colls)
        for _ in range(r.randrange(1, 3)):
            g = ctx.build(c.data, c.offsets)
            launches += ctx.last_build_stats()["graph"] > 0
            kept.append((g, want))
        what = r.randrange(8)
        if what == 0:  # the graph goes, its grammar stays
            ctx.set_graph(False)
            ctx.set_graph(True)
        elif what == 1:  # and the context
            ctxs.remove(ctx)
            other = r.choice(ctxs) if ctxs else None
            mine = [x for x in kept if x[0].ctx is ctx]
            kept = [x for x in kept if x[0].ctx is not ctx]
            ctx.close()
            if other is not None:
                for g, w in mine:
                    g.ctx = other
                    assert O.grammars_equal(g.export(), w), step
            for g, _ in mine:
                g.free()
        for g, w in kept:
            assert O.grammars_equal(g.export(), w), step
        while len(kept) > 3 or (kept and r.random() < 0.5):
            kept.pop(r.randrange(len(kept)))[0].free()
    assert launches > 100
