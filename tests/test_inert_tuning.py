"""A tuning field without effect is not searched, and changing it keeps a captured graph."""
import numpy as np
import pytest

import lcg_inputs as li
from paper_2411_12439_gb300 import autotune


class FakeCtx:
    INERT_TUNING = frozenset({"miss_flush"})

    def __init__(self):
        self.t = {"miss_flush": 64, "table_load": 0.35}
        self.seen = []

    def tuning(self):
        return dict(self.t)

    def set_tuning(self, **kw):
        self.t = dict(kw)
        self.seen.append(kw["miss_flush"])

    def build(self, data, offsets):
        return type("G", (), {"free": lambda self: None})()


def test_not_searched(monkeypatch):
    times = iter(range(1000, 0, -1))  # every trial beats the one before
    monkeypatch.setattr(autotune, "_time_builds", lambda *a: float(next(times)))
    ctx = FakeCtx()
    rep = autotune.autotune(ctx, None, None, reps=1)
    assert set(ctx.seen) == {64} and rep["tuning"]["miss_flush"] == 64
    assert all(t["miss_flush"] == 64 for t, _ in rep["trials"])


@pytest.mark.gpu
def test_graph_is_kept(hf):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_12439_gb300 import Context
    assert Context.INERT_TUNING == {"miss_flush"}
    coll = li.tiny_dna_collection(base_len=400_000, k=3)
    d = torch.from_numpy(np.ascontiguousarray(coll.data)).cuda()
    ctx = Context(hf, device=0)
    ctx.set_graph(True)
    modes = []
    for flush in (64, 64, 64, 128, 32):
        ctx.set_tuning(miss_flush=flush)
        ctx.build(d, coll.offsets).free()
        modes.append(ctx.last_build_stats()["graph"])
    assert modes[2:] == [2, 2, 2], modes
