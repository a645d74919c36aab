"""The all-pairs kernel's choice of lanes, clusters and cluster size, compiled
for the host: for every size, lane setting and memory budget it ends with an
answer, and a shape that it takes fits the memory and the GPU.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "shape.h"
using namespace bcm;
int main() {
    const uint32_t edge[] = {2, 63, 64, 65, 9727, 9728, 16384, 65536, 130000, 284000, 300000, 1064960, 1400000, 2129920,
                             4259840, 4260000, 5000000, 1u << 26, (1u << 30) - 1};
    long taken = 0, left = 0;
    for (int sms : {1, 8, 132, 152})
        for (size_t budget : {(size_t)0, (size_t)4096, (size_t)30 << 20, (size_t)64 << 20, (size_t)130 << 20})
            for (int lanes : {0, 64, 128, 256})
                for (uint64_t x = 0; x < 19 + 400; ++x) {
                    const uint32_t n = x < 19 ? edge[x] : (uint32_t)(2 + (x * x * x * 7919) % 6000000);
                    int W = -1, C = -1, k = -1;
                    if (!allpairs_fits(n, sms, budget, lanes, &W, &C, &k)) { ++left; continue; }
                    ++taken;
                    const bool ok = (W == 1 || W == 2 || W == 4) && (C == 1 || C == 2 || C == 4 || C == 8) && k >= 1 &&
                                    k * C <= sms && (size_t)k * allpairs_slot_bytes(n, W) <= budget &&
                                    (!lanes || lanes == 64 * W) && (uint64_t)(k - 1) * 64 * W < n;
                    if (!ok) { std::printf("n %u sms %d budget %zu lanes %d: W %d C %d clusters %d\n", n, sms, budget, lanes, W, C, k); return 1; }
                }
    std::printf("%ld %ld\n", taken, left);
    return 0;
}
"""


def test_every_size_gets_an_answer(tmp_path):
    src, exe = tmp_path / "shape.cc", tmp_path / "shape"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1507_01490_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, (res.returncode, res.stdout)   # (a division by zero ends it by a signal on x86)
    taken, left = map(int, res.stdout.split())
    assert taken > 1000 and left > 1000


def test_spread_steps(tmp_path):
    """i * spread_step(count) mod count visits every number below count once."""
    src, exe = tmp_path / "step.cc", tmp_path / "step"
    src.write_text('#include <cstdio>\n#include <vector>\n#include "shape.h"\n'
                   'int main() {\n'
                   '    for (uint32_t c = 1; c <= 4500; ++c) {\n'
                   '        std::vector<char> seen(c);\n'
                   '        const uint64_t s = bcm::spread_step(c);\n'
                   '        for (uint32_t i = 0; i < c; ++i) if (seen[i * s % c]++) { std::printf("%u\\n", c); return 1; }\n'
                   '    }\n'
                   '    return 0;\n}\n')
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1507_01490_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
