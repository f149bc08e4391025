"""The records of a timed build: one launch for all short rounds, whose further rounds
are marked as its own."""
import pytest

import lcg_inputs as li

pytestmark = pytest.mark.gpu


def test_short_rounds_share_one_launch(hf):
    from paper_2411_12439_gb300 import Context
    coll = li.tiny_dna_collection(base_len=400_000, k=3)
    ctx = Context(hf, device=0)
    for _ in range(2):  # round by round, then planned
        ctx.set_kernel_timing(1)
        ctx.build(coll.data, coll.offsets).free()
        rounds = ctx.last_build_stats()["rounds"]
        recs = ctx.last_kernel_launches()
        small = [r for r in recs if r["name"] == "k_parse_small"]
        assert [r["shared"] for r in small] == [False] + [True] * (len(small) - 1)
        assert small[0]["ms"] > 0 and all(r["ms"] == 0 and r["bytes"] == 0 for r in small[1:])
        parsed = [r["round"] for r in recs if r["name"] in ("k_parse", "k_parse_small")]
        assert parsed == list(range(1, rounds + 1))
        assert not any(r["shared"] for r in recs if r["name"] != "k_parse_small")


def test_last_rounds_share_one_launch_whatever_the_tile(hf):
    from paper_2411_12439_gb300 import Context
    coll = li.tiny_dna_collection(base_len=400_000, k=3)
    ctx = Context(hf, device=0)
    ctx.set_tuning(parse_tile=4096, parse_tile_min=0)
    for _ in range(2):
        ctx.set_kernel_timing(1)
        ctx.build(coll.data, coll.offsets).free()
        rounds = ctx.last_build_stats()["per_round"]
        small = [r["round"] for r in ctx.last_kernel_launches() if r["name"] == "k_parse_small"]
        assert small == [i + 1 for i, r in enumerate(rounds) if i + 1 >= small[0]]
        assert rounds[small[0] - 1]["n"] <= 1024 or rounds[small[0]]["n"] <= 1024
