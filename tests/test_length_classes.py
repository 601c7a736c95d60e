"""Host check of the fold-in schedule's length classes: inside the counters for
any 64-bit length, never later for a longer document, and the three groups
apart.  A small host program compiled with nvcc against the library's own
header; no GPU is used."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1704_03581_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "pulda_internal.h"
using namespace pulda;

int main() {
    int bad = 0;
    const int64_t coop[] = {1, 256, 300, 65535, 65536, INT64_MAX};
    for (int64_t c : coop) {
        auto check = [&](int64_t n) {
            const int x = length_class(n, c);
            const int lo = n > kNarrowMaxLen ? 0 : n >= c ? 1 : 1 + kLengthKeys;
            const int hi = n > kNarrowMaxLen ? 0 : n >= c ? kLengthKeys : 2 * kLengthKeys;
            if (x < lo || x > hi || x >= kLengthClasses) { std::printf("length %lld: class %d\n", static_cast<long long>(n), x); ++bad; }
        };
        int last = kLengthClasses;
        for (int64_t n = 0; n <= (int64_t(1) << 17); ++n) {
            check(n);
            if (length_class(n, c) > last) { std::printf("length %lld comes after a shorter one\n", static_cast<long long>(n)); ++bad; }
            last = length_class(n, c);
        }
        for (int s = 0; s < 64; ++s)
            for (int64_t d : {-1, 0, 1}) {
                const int64_t x = static_cast<int64_t>((uint64_t(1) << s) + static_cast<uint64_t>(d));
                check(x);
                check(static_cast<int64_t>(0 - static_cast<uint64_t>(x)));
            }
    }
    std::printf("violations %d\n", bad);
    return bad != 0;
}
"""


def test_length_classes_stay_inside_the_counters(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "classes.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "classes"
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and "violations 0" in out.stdout, out.stdout + out.stderr
