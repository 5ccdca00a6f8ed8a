"""What a device is asked once is asked once for every device (per_device.h, compiled for the
host: the answers come from functions of the test, no GPU takes part).
"""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1606_00548_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
static PerDevice a, b;
static std::atomic<int> asked{0};
static int ask(PerDevice &p, int dev, int answer) { return p.get(dev, [&] { asked++; return answer; }); }
int main() {
    for (int r = 0; r < 3; r++) {              // every device has its own answer, 0 among them
        if (ask(a, 0, 16) != 16 || ask(a, 1, 8) != 8 || ask(a, 2, 0) != 0 || ask(b, 0, 1) != 1) return 1;
        if (asked != 4) return 2;              // and is asked once
    }
    if (ask(a, -1, 3) != 3 || ask(a, 1000, 4) != 4 || ask(a, 1000, 5) != 5) return 3;   // outside: asked each time
    asked = 0;
    std::vector<std::thread> ts;
    std::atomic<int> wrong{0};
    for (int t = 0; t < 8; t++)
        ts.emplace_back([&] { for (int d = 3; d < 60; d++) if (ask(a, d, d) != d) wrong++; });
    for (auto &t : ts) t.join();
    return wrong != 0 ? 4 : asked < 57 || asked > 8 * 57 ? 5 : 0;
}
"""


def test_one_answer_per_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_no_kernel_attribute_is_set_under_a_plain_static():
    """every cudaFuncSetAttribute lies in a function that a PerDevice asks, or sets at each call"""
    import re
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"static\s+(const\s+)?(bool|int)\s+\w+\s*=\s*([^;]*);", text):
            assert "cudaFuncSetAttribute" not in m.group(3) and "_ctas(" not in m.group(3) and "[] {" not in m.group(3), (f, m.group(0)[:80])
