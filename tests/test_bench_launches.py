"""The benchmark's breakdown counts launches, not the rounds that share one, and gives the
time of a shared launch to its first round alone."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


class FakeCtx:
    def set_kernel_timing(self, mode):
        pass

    def build(self, d, offsets):
        return type("G", (), {"free": lambda self: None})()

    def last_build_stats(self):
        row = {"n": 8, "phrases": 4, "g": 2, "G": 4, "table_cap": 16, "strings": 1}
        return {"per_round": [dict(row) for _ in range(5)]}

    def last_kernel_launches(self):
        def rec(name, rnd, ms, shared=False):
            return {"name": name, "round": rnd, "ms": ms, "bytes": 0.0, "shared": shared}
        return [rec("k_breaks", 1, 0.5), rec("k_parse", 1, 2.0), rec("k_parse", 2, 1.0), rec("k_parse_small", 3, 0.25),
                rec("k_parse_small", 4, 0.0, True), rec("k_parse_small", 5, 0.0, True), rec("k_naming_small", 3, 0.125)]


def test_shared_launches():
    rounds, kernels = bench.round_breakdown(FakeCtx(), None, None)
    assert {k: v["launches"] for k, v in kernels.items()} == {"k_breaks": 1, "k_parse": 2, "k_parse_small": 1,
                                                              "k_naming_small": 1}
    assert [r["ms"] for r in rounds] == [2.5, 1.0, 0.375, None, None]
    assert [r["ms_rounds"] for r in rounds] == [1, 1, 3, 1, 1]
