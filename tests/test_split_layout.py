"""Host checks of the shared memory of documents on CTAs above 8,192 topics, for
every K the library accepts there: areas aligned, apart and within what a CTA
can have, and the chunks of the warps a partition of every lane's.  A small
host program compiled with nvcc against the library's own headers; no GPU is
used."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1704_03581_gb300", "csrc")

PROGRAM = r"""
#include <cstddef>
#include <cstdio>
#include "zsplit.cuh"
using namespace pulda;

static int bad = 0;
#define CHECK(cond, ...) do { if (!(cond)) { if (bad < 20) { std::printf(__VA_ARGS__); std::printf("\n"); } ++bad; } } while (0)

int main() {
    CHECK(offsetof(SplitCtl, part) % 16 == 0 && kSplitMapOff % 16 == 0, "control block");
    CHECK(kSplitMapOff >= static_cast<int>(sizeof(SplitCtl)) && kSplitColOff == kSplitMapOff + kMaxK / 8, "bits");
    CHECK(kSplitRecOff == kSplitColOff + 2 * 6 * kSplitColumn && kSplitCountOff == kSplitRecOff + 64 * (32 + 4), "columns and records");
    for (int K = kChainMaxK + 1; K <= kMaxK; ++K) {
        const int C = (K + 511) / 512, pb = 512 * C, rb = dense_row_bytes(K);
        CHECK(rb == 3 * pb && pb % 16 == 0 && (16 * C * 32) >= K, "K=%d: row", K);
        CHECK(split_smem_bytes(K) == kSplitCountOff + 3 * pb + 3 * rb && split_smem_bytes(K) <= 227 * 1024, "K=%d: %d bytes", K, split_smem_bytes(K));
        const int per = (C + kSplitWarps - 1) / kSplitWarps;
        int next = 0;
        for (int w = 0; w < kSplitWarps; ++w) {
            const int c0 = w * per < C ? w * per : C, c1 = c0 + per < C ? c0 + per : C;
            CHECK(c0 == next && c1 - c0 <= 8, "K=%d: warp %d has chunks %d to %d", K, w, c0, c1);
            next = c1;
        }
        CHECK(next == C, "K=%d: %d of %d chunks", K, next, C);
        CHECK(bitmap_row_words(K) <= kSplitMapWords && bitmap_row_words(K) % 4 == 0, "K=%d: bitmap row", K);
    }
    // the chain with three count planes
    for (int K = 1; K <= kChainMaxK; ++K) {
        const int ring = chain_ring_off(K, 3), pb = 128 * dense_words(K);
        CHECK(ring % 16 == 0 && kChainCountOff + 3 * chain_count_sets(K) * pb + (K > 1024 ? 64 * ((K + 511) / 512) : 0) <= ring, "K=%d: ring at %d", K, ring);
        CHECK(chain_smem_bytes(K, 3) == ring + 3 * chain_group(K) * 3 * pb && chain_smem_bytes(K, 3) <= 227 * 1024, "K=%d: %d bytes", K, chain_smem_bytes(K, 3));
        CHECK(chain_smem_bytes_upto(K, 3) >= chain_smem_bytes(K, 3), "chains up to K=%d", K);
    }
    std::printf("violations %d\n", bad);
    return bad != 0;
}
"""


def test_split_layout_stays_inside_its_buffers(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "split.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "split"
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr", "-I", CSRC,
                        "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and "violations 0" in out.stdout, out.stdout + out.stderr
