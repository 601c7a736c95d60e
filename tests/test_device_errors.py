"""Host check of what the error word of a chain's counters is reported as: every
bit has a status and a message of its own, a copy that did not arrive is not
called a grid barrier, and no bit is success.  A small host program compiled
with nvcc against the library's own headers; no GPU is used."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1704_03581_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "handle.h"
using namespace pulda;

int main() {
    const unsigned long long bits[] = {ERR_DEGENERATE, ERR_INTERNAL, ERR_GAMMA, ERR_BOUNDS, ERR_BARRIER, ERR_COPY};
    int bad = device_error(0).status != PULDA_OK;
    for (unsigned long long a : bits) {
        const DeviceError e = device_error(a);
        if (e.status == PULDA_OK || !e.message[0]) { std::printf("bit %llu: no error\n", a); ++bad; }
        for (unsigned long long b : bits)
            if (a != b && (a & b || !std::strcmp(e.message, device_error(b).message))) { std::printf("bits %llu, %llu\n", a, b); ++bad; }
    }
    const DeviceError copy = device_error(ERR_COPY);
    if (copy.status != PULDA_ERR_TIMEOUT || std::strstr(copy.message, "barrier")) { std::printf("copy: %s\n", copy.message); ++bad; }
    // what follows from a copy that failed does not hide it
    if (std::strcmp(device_error(ERR_COPY | ERR_INTERNAL).message, copy.message)) { std::printf("copy hidden\n"); ++bad; }
    std::printf("violations %d\n", bad);
    return bad != 0;
}
"""


def test_every_error_bit_has_its_own_message(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "errors.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "errors"
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and "violations 0" in out.stdout, out.stdout + out.stderr
