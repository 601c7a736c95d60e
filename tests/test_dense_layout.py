"""Host checks of the dense rows' index arithmetic, for every K the library
accepts: each topic's byte inside its plane and none shared, a lane's topics
where the kernels load them, the bitmap words a lane reads inside the row, and
the shared-memory areas of the one-warp and the long-document kernels aligned,
apart and within what a CTA can have.  A small host program compiled with nvcc
against the library's own headers prints any violation; no GPU is used."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1704_03581_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdint>
#include <vector>
#include "zchain.cuh"
using namespace pulda;

static int bad = 0;
#define CHECK(cond, ...) do { if (!(cond)) { if (bad < 20) { std::printf(__VA_ARGS__); std::printf("\n"); } ++bad; } } while (0)

int main() {
    for (int K = 1; K <= kMaxK; ++K) {
        const int nw = dense_words(K), tpl = 4 * nw, pb = 128 * nw, C = (K + 511) / 512;
        CHECK(32 * tpl >= K, "K=%d: %d topics per lane", K, tpl);
        CHECK(z_nw(K) == 0 || z_nw(K) == 1 || z_nw(K) == 2 || z_nw(K) == 4 || z_nw(K) == 8, "K=%d: form %d", K, z_nw(K));
        CHECK(z_nw(K) == 0 ? nw == 4 * C : nw == z_nw(K), "K=%d: %d words", K, nw);
        CHECK(dense_row_bytes(K) == 3 * pb && pb % 16 == 0, "K=%d: row", K);
        std::vector<char> seen(pb, 0);
        const uint32_t recip = static_cast<uint32_t>((0x100000000ull + tpl - 1) / tpl);
        for (int k = 0; k < K; ++k) {
            const int p = dense_pos(K, k), l = k / tpl, b = k % tpl;
            CHECK(p >= 0 && p < pb && !seen[p], "K=%d: topic %d at %d", K, k, p);
            if (p >= 0 && p < pb) seen[p] = 1;
            // where a lane's loads find it: up to 512 topics consecutive bytes, above chunks of 16
            CHECK(p == (K <= 512 ? tpl * l + b : (b >> 4) * 512 + 16 * l + (b & 15)), "K=%d: topic %d of lane %d", K, k, l);
            if (K > 1024) {
                CHECK(static_cast<int>((static_cast<uint64_t>(k) * recip) >> 32) == l, "K=%d: lane of %d", K, k);
                CHECK(((p >> 4) & 31) * tpl + ((p >> 9) << 4) + (p & 15) == k, "K=%d: topic at %d", K, p);
            } else if (K > 512) {
                CHECK((((p & 512) >> 5) | ((p & 496) << 1) | (p & 15)) == k, "K=%d: topic at %d", K, p);
                CHECK((((k & 16) << 5) | ((k >> 5) << 4) | (k & 15)) == p, "K=%d: position of %d", K, k);
            }
        }
        // a lane's bits: one word (K <= 1024), C half words above
        const int words = bitmap_row_words(K);
        CHECK(32 * words >= K && words % 4 == 0, "K=%d: bitmap row of %d", K, words);
        if (K <= 1024) CHECK(((31 * tpl) >> 5) < words, "K=%d: lane 31 reads word %d", K, (31 * tpl) >> 5);
        else CHECK(32 * C <= 2 * words, "K=%d: half word %d of %d", K, 32 * C - 1, 2 * words);
        for (bool narrow : {true, false}) {
            const int w = z_dense_count_words(K, narrow);
            CHECK(w % 4 == 0 && z_dense_warp_words(K, narrow) % 4 == 0, "K=%d: areas not 16-byte aligned", K);
            CHECK(4 * w >= z_count_planes(narrow) * pb + (K > 1024 ? 64 * C : 0), "K=%d: counts", K);
            CHECK(4 * z_dense_warp_words(K, narrow) <= 227 * 1024, "K=%d: a warp's area", K);
        }
        const int G = chain_group(K), ring = chain_ring_off(K);
        CHECK(G >= 1 && G <= 8 && 32 % G == 0, "K=%d: groups of %d", K, G);
        CHECK(ring % 16 == 0 && kChainCountOff + 2 * chain_count_sets(K) * pb + (K > 1024 ? 64 * C : 0) <= ring, "K=%d: ring at %d", K, ring);
        CHECK(chain_smem_bytes(K) == ring + 3 * G * 3 * pb && chain_smem_bytes(K) <= 227 * 1024, "K=%d: %d bytes", K, chain_smem_bytes(K));
    }
    int most = 0;
    for (int K = 1; K <= kMaxK; ++K) {
        most = chain_smem_bytes(K) > most ? chain_smem_bytes(K) : most;
        CHECK(chain_smem_bytes_upto(K) >= most, "chains up to K=%d: %d of %d bytes", K, chain_smem_bytes_upto(K), most);
    }
    std::printf("violations %d\n", bad);
    return bad != 0;
}
"""


def test_dense_rows_stay_inside_their_buffers(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "layout.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "layout"
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr", "-I", CSRC,
                        "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and "violations 0" in out.stdout, out.stdout + out.stderr
