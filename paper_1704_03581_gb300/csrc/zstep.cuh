// What the z-step kernels share (kernels.cu: one warp per document; coop.cu:
// one CTA per document; zgroup.cu: four documents per warp): the per-document
// run, the staging of a token's token-only data, the warp's counters and the
// shared-memory sizes.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

#include "device_rng.cuh"
#include "pulda_internal.h"
#include "checks.cuh"

namespace pulda {

typedef unsigned long long u64;

__device__ __forceinline__ u64 warp_sum64(u64 v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

__device__ __forceinline__ uint32_t sweep_of(const ZArgs &a) { return a.sweep_ptr ? *a.sweep_ptr : a.sweep; }

// Layout of a count array with a gap word after every lane's topics and a
// leading zero (32- or 16-bit counts), whose arithmetic has host checks of its
// own; the kernels hold counts as planes of bytes (z_dense_count_words).
__host__ __device__ __forceinline__ int mi(int k) { return k + (k >> 5); }
__host__ __device__ __forceinline__ int z_lane_topics(int K) {
    return K <= 256 ? 8 : K <= 512 ? 16 : K <= 1024 ? 32 : 64;
}
__host__ __device__ __forceinline__ int z_m_words(int K) { return (K + (K >> 5) + 32 + 1 + 3) & ~3; }
template <typename CT>
__host__ __device__ __forceinline__ int z_count_words(int K) {
    return sizeof(CT) == 4 ? z_m_words(K) : ((K + (K >> 5) + 32 + 2 + 1) / 2 + 3) & ~3;
}

constexpr int kTokRecWords = 9;     // two uint4 per token, and its word's dense row
// A warp's six 64-bit counters (16-byte aligned) and the document run it is
// working on: {tokens, alias draws, sum min(K_d, K_v), zero-mass tokens,
// sum |J|, tokens with K_d < K_v}, lane j updating counter j.
constexpr int kWarpCountWords = 32;

// One document's run: where its tokens live and where its Markov chain is.
struct DocRun {
    const int32_t *w;        // word ids, position 0 first
    int16_t *z;              // topics, updated in place
    int len;
    uint64_t seed;
    int64_t index_base;      // RNG index of position 0
    uint32_t sweep;          // sweep counter of the pass that starts at `pos`
    int pos;                 // first position to resample
    int64_t budget;          // tokens to resample in this call (passes continue past the end)
    int max_pass_end;        // stop when the pass counter reaches sweep + this many passes
    uint64_t deadline = ~0ull;   // global timer (ns): no 32-token block starts after it, but the first
};
// The run a z-step warp is working on, kept after its six counters (8-byte
// aligned: the counter area starts 16-byte aligned).
static_assert(6 * sizeof(unsigned long long) + sizeof(DocRun) <= kWarpCountWords * sizeof(uint32_t),
              "the warp's counters and document run must fit its counter area");
__device__ __forceinline__ DocRun *z_warp_run(unsigned long long *wcnt) { return reinterpret_cast<DocRun *>(wcnt + 6); }


__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The alias draw of the a part (Walker): slot e of the word's column keeps its
// own topic when the uniform u is below the slot's threshold, else takes the
// slot's alias topic.  Read from the packed slots when the tables carry them.
__device__ __forceinline__ int alias_outcome(const ZArgs &a, int64_t e, uint32_t u) {
    if (a.apack) {
        const uint2 s = a.apack[e];
        return guard_index(static_cast<int>(u < s.x ? s.y & 0xFFFFu : s.y >> 16), a.K, a.stats);
    }
    return guard_index(u < a.athr[e] ? a.topic[e] : a.atopic[e], a.K, a.stats);
}

// What depends only on a token, gathered in three steps that each wait for the
// loads of the one before: its word, topic and Philox words; its word's
// column, sigma_a and dense row (~0 when it is to be summed over its column: it
// has at most colmax topics, or no row); its alias outcome.
struct StagedToken {
    int word, topic;
    U4 x;
    int64_t col;
    int n_w;
    u64 A;
    uint32_t row;
    __device__ __forceinline__ void load_token(const ZArgs &a, const DocRun &r, int i) {
        word = r.w[i];
        topic = guard_index(r.z[i], a.K, a.stats);
        const uint64_t t = static_cast<uint64_t>(r.index_base + i);
        x = draw(r.seed, static_cast<uint32_t>(t), static_cast<uint32_t>(t >> 32), r.sweep, TAG_Z, 0);
    }
    __device__ __forceinline__ void load_word(const ZArgs &a, int colmax) {
        col = a.col_ptr[word];
        n_w = static_cast<int>(a.col_ptr[word + 1] - col);
        A = a.A[word];
        const uint32_t d = static_cast<uint32_t>(a.drow[word]);
        row = n_w > colmax ? d : 0xFFFFFFFFu;
    }
    __device__ __forceinline__ int load_alias(const ZArgs &a) const {
        return n_w > 0 ? alias_outcome(a, col + __umulhi(x.z, static_cast<uint32_t>(n_w)), x.w) : 0;
    }
};

// Stages token i of run r for the one-warp kernel,
//   rec2[0] = {column start (low 32), column start >> 32 | alias outcome << 16, sigma_a (lo, hi)}
//   rec2[1] = {Philox x0, x1, word, K_v | old topic << 16}
// and its dense row.  Topics are staged as their positions, pos(k) (column
// starts are below 2^48, K_v <= 16384, positions < 16384).
template <typename Pos>
__device__ __forceinline__ void stage_token(const ZArgs &a, const DocRun &r, int i, uint4 *rec2, uint32_t *drow, int colmax, Pos pos) {
    StagedToken s;
    s.load_token(a, r, i);
    s.load_word(a, colmax);
    const int ta = pos(s.load_alias(a));
    rec2[0] = make_uint4(static_cast<uint32_t>(s.col),
                         static_cast<uint32_t>(static_cast<u64>(s.col) >> 32) | (static_cast<uint32_t>(ta) << 16),
                         static_cast<uint32_t>(s.A), static_cast<uint32_t>(s.A >> 32));
    rec2[1] = make_uint4(s.x.x, s.x.y, static_cast<uint32_t>(s.word),
                         static_cast<uint32_t>(s.n_w) | (static_cast<uint32_t>(pos(s.topic)) << 16));
    *drow = s.row;
}


// Shared memory of a z-step warp on dense rows, in 32-bit words: the count
// planes (two, or three when a document may have 2^16 tokens or more), above
// 1024 topics the lanes' 16 bits per chunk of nonzero topics, the staging
// records, the counters and the run.
__host__ __device__ __forceinline__ int z_nw(int K) { return K <= 1024 ? dense_words(K) : 0; }    // the form of z_doc
__host__ __device__ __forceinline__ int z_count_planes(bool narrow) { return narrow ? 2 : 3; }
__host__ __device__ __forceinline__ int z_dense_count_words(int K, bool narrow) {
    return 32 * dense_words(K) * z_count_planes(narrow) + (K > 1024 ? 4 * dense_words(K) : 0);
}
__host__ __device__ __forceinline__ int z_dense_warp_words(int K, bool narrow) {
    return z_dense_count_words(K, narrow) + 32 * kTokRecWords + kWarpCountWords;
}
__device__ __forceinline__ unsigned long long *z_dense_counters(uint32_t *sm, int K, bool narrow) {
    return reinterpret_cast<unsigned long long *>(sm + z_dense_count_words(K, narrow) + 32 * kTokRecWords);
}

// A lane's TPL bits of a bitmap row starting at word `row` (TPL <= 32).
template <int TPL>
__device__ __forceinline__ uint32_t lane_bits(const uint32_t *bits, int64_t row, int lane) {
    if constexpr (TPL == 32) {
        return bits[row + lane];
    } else {
        const uint32_t w = bits[row + (lane * TPL >> 5)];
        return (w >> ((lane * TPL) & 31)) & ((1u << (TPL & 31)) - 1u);
    }
}

// Zeroes, and adds to the sweep's and the running totals, a warp's counters
// kept in its shared memory.  Every lane calls them.
__device__ __forceinline__ void zero_warp_counters(unsigned long long *cnt) {
    if ((threadIdx.x & 31) < 6) cnt[threadIdx.x & 31] = 0;
    __syncwarp();
}

__device__ inline void flush_warp_counters(unsigned long long *stats, unsigned long long *cnt) {
    const int lane = threadIdx.x & 31;
    // lane j's counter goes to slot {tokens, a-branch, sum min, zero mass, sum |J|, doc side}[j]
    const int slot = lane == 0 ? ST_TOKENS : lane == 1 ? ST_ABRANCH : lane == 2 ? ST_SUMMIN
                   : lane == 3 ? ST_ZEROMASS : lane == 4 ? ST_SUMINT : ST_DOCSIDE;
    __syncwarp();
    if (lane < 6) {
        const unsigned long long v = cnt[lane];
        if (v) {
            atomicAdd(&stats[slot], v);
            atomicAdd(&stats[ST_COUNT + slot], v);
        }
        cnt[lane] = 0;
    }
    __syncwarp();
}

// Opt a kernel in to the largest dynamic shared memory it can use next to
// its static shared memory.
template <typename F>
void allow_dynamic_smem(F *kernel) {
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) return;
    const int room = smem_optin() - static_cast<int>(fa.sharedSizeBytes);
    if (room > 0) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, room);
}

}  // namespace pulda
