"""What a launch asks of a device (shared memory limits, resident blocks) is kept per
device: csrc/per_device.h, compiled and run on the CPU with made-up devices, and no
launcher keeps such an answer for the whole process."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2411_12439_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
static lcg::PerDevice<int> known;
int main() {
    int calls[4] = {0}, bad = 0;
    auto ask = [&](int dev, int fail) {
        int v = -1;
        const int e = known.get(dev, v, [&](int& x) { calls[dev]++; x = 100 + dev; return fail; });
        return e ? -e : v;
    };
    bad += ask(0, 0) != 100 || ask(1, 0) != 101;   // each device's own value
    bad += ask(0, 7) != 100 || calls[0] != 1;       // made once
    bad += ask(2, 7) != -7 || ask(2, 0) != 102 || calls[2] != 2;  // a failure is reported and not kept
    std::vector<std::thread> ts;
    std::vector<int> got(16);
    for (int i = 0; i < 16; i++) ts.emplace_back([&, i] { got[i] = ask(3, 0); });
    for (auto& t : ts) t.join();
    for (int x : got) bad += x != 103;
    bad += calls[3] != 1;
    int v = 0, n = 0;
    for (int d : {-1, lcg::kMaxDevices}) known.get(d, v, [&](int& x) { n++; x = d; return 0; });
    bad += n != 2 || v != lcg::kMaxDevices;         // past the array: asked every time
    std::printf("%d\n", bad);
    return bad;
}
"""


def test_value_per_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-o", str(exe), str(src)])
    assert subprocess.run([str(exe)]).returncode == 0


def test_no_answer_of_one_device_is_kept_for_all():
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"\bstatic const\b[^;{]*=\s*(\[\]|cuda)", text):
            raise AssertionError(f"{f}: {text[m.start():m.end() + 60]!r}")
