// CUDA kernels of the Polya-urn partially collapsed LDA sampler, sm_103a.
//
// One sweep = Algorithm 2 (Section 3):
//   Phi-step  k_heavy_hist   the most frequent words histogrammed in chunks by
//                            many CTAs.
//             k_phi_counts   per word v: rebuild n_{.,v} from z (shared-memory
//                            histogram over the word's tokens), draw
//                            c_{k,v} ~ Pois(beta + n_{k,v}) for every k (Eq. 9,
//                            "Efficient sampling of Phi"), accumulate S_k.
//             k_phi_fixup    rows with S_k = 0 are redrawn until nonzero
//                            (Definition "Poisson Polya Urn").
//             k_scan         column offsets of the sparse Phi.
//             k_phi_tables   phi = c/S, fixed-point weights, sigma_a, the
//                            per-word alias table, bitmaps and dense q rows
//                            ("Efficient sampling of z").
//   z-step    k_z_step       one warp per document, tokens in order, the a/b
//                            draw over dense rows of weights (k_slice_counts first
//                            when long documents run in stale-count slices).
// The *_multi kernels do the same over many chains; k_serve_step folds in
// requests; k_z_step_pairs takes two documents per warp; the longest documents
// go to CTAs of their own (coop.cu); Algorithm 1's Dirichlet Phi-step is in dirichlet.cu.
// The arithmetic that decides any draw is integer or IEEE double with
// explicit rounding (or integers that give the double's value), so results are independent of launch shapes.
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <type_traits>

#include "device_rng.cuh"
#include "pulda_internal.h"
#include "zdense.cuh"
#include "zpair.cuh"
#include "zstep.cuh"
#include "checks.cuh"

namespace pulda {
namespace {



// ------------------------------------------------------- Phi-step draws
// Alias-table draw from table t: slot floor(xs * n / 2^32), kept if xa < thr.
__device__ __forceinline__ uint32_t table_draw(const DevTables &T, int t, uint32_t xs, uint32_t xa) {
    const int off = T.off[t];
    const uint32_t s = __umulhi(xs, static_cast<uint32_t>(T.n[t]));
    const uint32_t j = xa < T.thr[off + s] ? s : static_cast<uint32_t>(T.alias[off + s]);
    return static_cast<uint32_t>(T.lo[t] + static_cast<int>(j));
}

// c ~ Pois(beta + l) for l >= 1: alias table for l <= L, rounded Gaussian
// mu + sqrt(mu) g, mu = beta + l, above.  g is interpolated linearly inside
// one of 2^16 equiprobable cells of the normal law.
__device__ uint32_t draw_entry(const DevTables &T, uint32_t l, uint32_t x0, uint32_t x1) {
    if (l <= static_cast<uint32_t>(kL)) return table_draw(T, static_cast<int>(l), x0, x1);
    const double g = gauss_draw(T, x0, x1);
    const double mu = __dadd_rn(T.beta, static_cast<double>(l));
    const double sd = __dsqrt_rn(mu);
    double r = floor(__dadd_rn(__dadd_rn(mu, __dmul_rn(sd, g)), 0.5));
    if (r < 0.0) r = 0.0;
    if (r > 4294967295.0) r = 4294967295.0;
    return static_cast<uint32_t>(r);
}

// Smallest g with x < geo[g]; -1 when the gap is at least kGeoLen.
__device__ __forceinline__ int geo_gap(const uint32_t *geo, uint32_t x) {
    if (x >= geo[kGeoLen - 1]) return -1;
    int lo = 0, hi = kGeoLen - 1;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (x < geo[mid]) hi = mid; else lo = mid + 1;
    }
    return lo;
}

// ------------------------------------------------------- block helpers
template <int BLOCK>
__device__ __forceinline__ int block_excl_scan(int v, int *tmp /* >= BLOCK/32 + 1 */, int &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) tmp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int t = lane < BLOCK / 32 ? tmp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < BLOCK / 32) tmp[lane] = t;
    }
    __syncthreads();
    total = tmp[BLOCK / 32 - 1];
    const int base = warp ? tmp[warp - 1] : 0;
    __syncthreads();
    return base + x - v;
}

// ================================================================= init
__global__ void k_init_z(int64_t N, int K, uint64_t seed, int64_t base, int16_t *z) {
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < N;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const uint64_t t = static_cast<uint64_t>(base + i);
        const U4 x = draw(seed, static_cast<uint32_t>(t), static_cast<uint32_t>(t >> 32), 0, TAG_INIT, 0);
        z[i] = static_cast<int16_t>(__umulhi(x.x, static_cast<uint32_t>(K)));
    }
}

// word-major permutation: counting sort of token ids by word id
__global__ void k_word_hist(int64_t N, const int32_t *w, int32_t *cnt) {
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < N;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        atomicAdd(&cnt[w[i]], 1);
}

// Exclusive scan of cnt[0..n) into out[0..n] (out[n] = total), chunk by chunk
// of the entries: a CTA adds up everything before its chunk itself, so the
// chunks wait neither for each other nor for a second launch.  The repeated
// reads come from L2 (400 KB for 100,000 words); one CTA over all the entries,
// each thread over a stretch of its own, was bound by its uncoalesced loads:
// 106 us for 100,000 words, the chunks take 12.
constexpr int kScanChunk = 2048;
__host__ __device__ __forceinline__ int64_t scan_chunk(int64_t n) {     // entries per CTA: at most 256 CTAs
    const int64_t c = (n + 255) / 256;
    return c <= kScanChunk ? kScanChunk : (c + 3) / 4 * 4;
}
__host__ __device__ __forceinline__ int scan_chunks(int64_t n) { return static_cast<int>(n > 0 ? (n + scan_chunk(n) - 1) / scan_chunk(n) : 1); }

template <int BLOCK>
__device__ void scan_one_chunk(const int32_t *cnt, int64_t n, int64_t *out, unsigned long long *total_slot, int c, int *tmp,
                               u64 *red) {
    const int64_t size = scan_chunk(n), lo = c * size, hi = min(n, lo + size);
    const int4 *c4 = reinterpret_cast<const int4 *>(cnt);
    u64 before = 0;
#pragma unroll 4
    for (int64_t i = threadIdx.x; i < lo / 4; i += BLOCK) {
        const int4 x = __ldcg(&c4[i]);
        before += static_cast<u64>(x.x) + static_cast<u64>(x.y) + static_cast<u64>(x.z) + static_cast<u64>(x.w);
    }
    before = warp_sum64(before);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = before;
    __syncthreads();
    int64_t run = 0;
    for (int i = 0; i < BLOCK / 32; ++i) run += static_cast<int64_t>(red[i]);
    for (int64_t t0 = lo; t0 < hi; t0 += 4 * BLOCK) {
        const int64_t t = t0 + 4 * threadIdx.x;
        int x[4] = {0, 0, 0, 0};
        if (t + 3 < hi) {
            const int4 y = __ldcg(&c4[t / 4]);
            x[0] = y.x; x[1] = y.y; x[2] = y.z; x[3] = y.w;
        } else {
            for (int j = 0; j < 4 && t + j < hi; ++j) x[j] = __ldcg(&cnt[t + j]);
        }
        int total;
        int64_t o = run + block_excl_scan<BLOCK>(x[0] + x[1] + x[2] + x[3], tmp, total);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (t + j < hi) out[t + j] = o;
            o += x[j];
        }
        run += total;
    }
    if (hi == n && threadIdx.x == 0) {
        out[n] = run;
        if (total_slot) *total_slot = static_cast<unsigned long long>(run);
    }
    __syncthreads();
}

constexpr int kScanBlock = 512;
__global__ void __launch_bounds__(kScanBlock) k_scan(const int32_t *cnt, int64_t n, int64_t *out, unsigned long long *total_slot) {
    __shared__ int tmp[kScanBlock / 32 + 1];
    __shared__ u64 red[kScanBlock / 32];
    scan_one_chunk<kScanBlock>(cnt, n, out, total_slot, blockIdx.x, tmp, red);
}

// Column offsets of every chain's Phi: chunk blockIdx.y of chain blockIdx.x.
__global__ void __launch_bounds__(kScanBlock) k_colptr_scan_multi(const PhiArgs *chains) {
    __shared__ int tmp[kScanBlock / 32 + 1];
    __shared__ u64 red[kScanBlock / 32];
    const PhiArgs &a = chains[blockIdx.x];
    if (static_cast<int>(blockIdx.y) >= scan_chunks(a.V)) return;
    scan_one_chunk<kScanBlock>(a.nnz_c, a.V, a.col_ptr, &a.stats[ST_NNZPHI], blockIdx.y, tmp, red);
}

__global__ void k_word_scatter(int64_t N, const int32_t *w, const int64_t *word_off, int32_t *fill, int32_t *perm) {
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < N;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int v = w[i];
        const int pos = atomicAdd(&fill[v], 1);
        perm[word_off[v] + pos] = static_cast<int32_t>(i);
    }
}

// ======================================================== Phi-step: counts
constexpr int kPhiBlock = 256;
#ifndef PULDA_PHI_COUNT_BLOCK
#define PULDA_PHI_COUNT_BLOCK 128
#endif
constexpr int kPhiCountBlock = PULDA_PHI_COUNT_BLOCK;

// Sweep counter of a chain: from device memory when the launch is replayed
// from a CUDA graph (one graph serves every sweep), else the launch value.
__device__ __forceinline__ uint32_t sweep_of(const PhiArgs &a) { return a.sweep_ptr ? *a.sweep_ptr : a.sweep; }

// Adds the topics of the word-ordered tokens [b, e) into hist (shared
// memory), by a CTA of BLOCK threads.  The topics are gathered through perm
// from all over the corpus, so each thread issues kHistBatch of those loads
// before the first atomic: latency, not bandwidth, bounds a loop that waits
// on one at a time.
#ifndef PULDA_HIST_BATCH
#define PULDA_HIST_BATCH 8
#endif
constexpr int kHistBatch = PULDA_HIST_BATCH;
template <int BLOCK>
__device__ __forceinline__ void hist_tokens(const PhiArgs &a, int64_t b, int64_t e, uint32_t *hist) {
    const int K = a.K;
    int64_t t = b + threadIdx.x;
    for (; t + (kHistBatch - 1) * BLOCK < e; t += kHistBatch * BLOCK) {
        int32_t p[kHistBatch];
        int zz[kHistBatch];
#pragma unroll
        for (int u = 0; u < kHistBatch; ++u) p[u] = a.perm[t + u * BLOCK];
#pragma unroll
        for (int u = 0; u < kHistBatch; ++u) zz[u] = a.z[p[u]];
#pragma unroll
        for (int u = 0; u < kHistBatch; ++u) atomicAdd(&hist[guard_index(zz[u], K, a.stats)], 1u);
    }
    for (; t < e; t += BLOCK) atomicAdd(&hist[guard_index(a.z[a.perm[t]], K, a.stats)], 1u);
}

// One word v of one chain, by the whole CTA of BLOCK threads: histogram of
// the word's topics -> n_{.,v}; compacted n column; when `draw`, the Poisson
// draws c_{.,v}, the compacted c column, and S_k += c_{k,v}.  hist/cbin hold
// K entries each.  With `next` set, thread 0 takes the CTA's next work item
// from `work` once every thread is past reading the current one; the last
// barrier publishes it.
template <int BLOCK>
__device__ void phi_word(const PhiArgs &a, int v, bool do_draw, uint32_t *hist, uint32_t *cbin, int *scan_tmp,
                         const uint32_t *geo, int *next = nullptr, int *work = nullptr) {
    const int K = a.K;
    const uint32_t sweep = sweep_of(a);
    const int per = (K + BLOCK - 1) / BLOCK;     // bins owned by each thread, contiguous
    const int64_t wbeg = a.word_off[v], wend = a.word_off[v + 1];
    const int hrow = a.heavy_row ? a.heavy_row[v] : -1;
    if (a.counted) {
        // the n column was built by the sort path (countsort.cu)
        for (int k = threadIdx.x; k < K; k += BLOCK) { hist[k] = 0; cbin[k] = 0; }
        __syncthreads();
        const int nn = a.nnz_n[v];
        for (int j = threadIdx.x; j < nn; j += BLOCK)
            hist[guard_index(a.nst_k[wbeg + j], K, a.stats)] = a.nst_n[wbeg + j];
        __syncthreads();
    } else if (hrow >= 0) {
        // from L2: just summed by other CTAs; left zero for the next time
        uint32_t *hh = a.heavy_hist + static_cast<int64_t>(hrow) * K;
        for (int k = threadIdx.x; k < K; k += BLOCK) { hist[k] = __ldcg(&hh[k]); hh[k] = 0; cbin[k] = 0; }
        __syncthreads();
    } else {
        for (int k = threadIdx.x; k < K; k += BLOCK) { hist[k] = 0; cbin[k] = 0; }
        __syncthreads();
        hist_tokens<BLOCK>(a, wbeg, wend, hist);
        __syncthreads();
    }
    if (next && threadIdx.x == 0) *next = atomicAdd(work, 1);
    if (do_draw) {
        // entries with n_{k,v} = l >= 1: c ~ Pois(beta + l)
        for (int k = threadIdx.x; k < K; k += BLOCK) {
            const uint32_t l = hist[k];
            if (l) {
                const U4 x = draw(a.seed, static_cast<uint32_t>(v), static_cast<uint32_t>(k), sweep, TAG_POIS, 0);
                cbin[k] = draw_entry(a.tab, l, x.x, x.y);
            }
        }
        // entries with n_{k,v} = 0: Pois(beta) by geometric skip-ahead.  The
        // walk's draws h = 0, 1, ... do not depend on where it stands, so
        // warp 0 draws 32 of them at once and a prefix sum of the gaps places
        // them -- the same hits, in the same order, as one thread walking.
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x;
            int pos = -1;
            for (uint32_t h0 = 0;; h0 += 32) {
                const U4 x = draw(a.seed, static_cast<uint32_t>(v), h0 + lane, sweep, TAG_BETA, 0);
                const int g = geo_gap(geo, x.x);
                const int step = g < 0 ? kGeoLen : g + 1;      // positions advanced by this draw
                int incl = step;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    if (lane >= o) incl += y;
                }
                const int p = pos + incl;                       // the hit's position (or where a skip ends)
                const bool stop = g < 0 ? p >= K - 1 : p >= K;
                const uint32_t bal = __ballot_sync(0xFFFFFFFFu, stop);
                const int first_stop = bal ? __ffs(bal) - 1 : 32;
                if (lane < first_stop && g >= 0 && hist[p] == 0) cbin[p] = table_draw(a.tab, 0, x.y, x.z);
                if (bal) break;
                pos = __shfl_sync(0xFFFFFFFFu, p, 31);
            }
        }
        __syncthreads();
    }
    // compaction in ascending topic order
    const int k0 = threadIdx.x * per, k1 = min(K, k0 + per);
    int cn = 0, cc = 0;
    for (int k = k0; k < k1; ++k) { cn += hist[k] != 0; cc += cbin[k] != 0; }
    // one scan of both counts, n's in the low and c's in the high 16 bits
    // (each at most K <= 16384)
    int tboth;
    const int pboth = block_excl_scan<BLOCK>(cn | (cc << 16), scan_tmp, tboth);
    int pn = pboth & 0xFFFF, pc = pboth >> 16;
    const int tn = tboth & 0xFFFF, tc = tboth >> 16;
    for (int k = k0; k < k1; ++k) {
        const uint32_t l = hist[k];
        if (l) { a.nst_k[wbeg + pn] = static_cast<uint16_t>(k); a.nst_n[wbeg + pn] = l; ++pn; }
        if (do_draw) {
            const uint32_t c = cbin[k];
            if (c) {
                const int64_t o = static_cast<int64_t>(v) * K + pc;
                a.cst_k[o] = static_cast<uint16_t>(k);
                a.cst_c[o] = c;
                atomicAdd(&a.S[k], static_cast<u64>(c));
                ++pc;
            }
        }
    }
    if (threadIdx.x == 0) {
        a.nnz_n[v] = tn;
        if (do_draw) a.nnz_c[v] = tc;
    }
    __syncthreads();
}

// A word of at most kWarpWord tokens, by one warp.  Most words are rare: a pass
// of a CTA over all K topics, several times with barriers in between, costs
// far more than the word's few entries.  pk[k] holds n_{k,v} in the low and
// c_{k,v} in the high 16 bits (n <= 256, so c ~ Pois(beta + n) stays far
// below 2^16), with bitmaps of the topics that have either.  A lane lists the
// topics of its bitmap words in ascending order, then the lanes share out the
// list, so the draws and the stores do not wait on the lane of the most topics.
// pk and the bitmaps are zero between words; kmax lays them out, the same for
// every word of a launch.  (100,000 words, 12.4 M tokens, K = 1000: the pass
// took 600 us with a CTA per word and 500 with these warps; the rest of the way
// to 200 is heavy_word's.  Limits of 64 to 1,024 tokens differ by less than the
// runs do.  K = 3000: 0.28 ms less; above 4,096 topics a CTA's warps no longer
// have room beside another CTA.)
constexpr int64_t kWarpWord = 256;
constexpr int kWarpWordMaxK = 4096;
__host__ __device__ __forceinline__ int warp_word_words(int K) {
    return ((K + 3) & ~3) + 2 * (((K + 31) / 32 + 3) & ~3) + (((K + 1) / 2 + 3) & ~3);
}

// The topics of a bitmap of KW words as a list, by one warp; returns how many.
__device__ __forceinline__ int list_topics(const uint32_t *bitmap, int KW, uint16_t *list) {
    const int lane = threadIdx.x & 31;
    int base = 0;
    for (int w0 = 0; w0 < KW; w0 += 32) {
        const int w = w0 + lane;
        uint32_t bits = w < KW ? bitmap[w] : 0u;
        int x = __popc(bits);
        const int own = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        uint16_t *o = list + base + x - own;
        for (; bits; bits &= bits - 1u) *o++ = static_cast<uint16_t>(32 * w + __ffs(bits) - 1);
        base += __shfl_sync(0xFFFFFFFFu, x, 31);
    }
    __syncwarp();
    return base;
}

__device__ void phi_word_warp(const PhiArgs &a, int v, bool do_draw, uint32_t *pk, int kmax, const uint32_t *geo) {
    const int lane = threadIdx.x & 31;
    const int K = a.K, KW = (K + 31) >> 5;
    const int kw_max = ((kmax + 31) / 32 + 3) & ~3;
    uint32_t *nb = pk + ((kmax + 3) & ~3), *cb = nb + kw_max;
    uint16_t *list = reinterpret_cast<uint16_t *>(cb + kw_max);
    const uint32_t sweep = sweep_of(a);
    const int64_t wbeg = a.word_off[v], wend = a.word_off[v + 1];
    auto add = [&](int k) {
        if (atomicAdd(&pk[k], 1u) == 0) atomicOr(&nb[k >> 5], 1u << (k & 31));
    };
    int64_t t = wbeg + lane;
    for (; t + 3 * 32 < wend; t += 4 * 32) {
        int p[4], zz[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) p[u] = a.perm[t + 32 * u];
#pragma unroll
        for (int u = 0; u < 4; ++u) zz[u] = a.z[p[u]];
#pragma unroll
        for (int u = 0; u < 4; ++u) add(guard_index(zz[u], K, a.stats));
    }
    for (; t < wend; t += 32) add(guard_index(a.z[a.perm[t]], K, a.stats));
    __syncwarp();
    // the n column, and c ~ Pois(beta + n) for its entries
    const int nn = list_topics(nb, KW, list);
    for (int i = lane; i < nn; i += 32) {
        const int k = list[i];
        const uint32_t l = pk[k];
        a.nst_k[wbeg + i] = static_cast<uint16_t>(k);
        a.nst_n[wbeg + i] = l;
        if (do_draw) {
            const U4 x = draw(a.seed, static_cast<uint32_t>(v), static_cast<uint32_t>(k), sweep, TAG_POIS, 0);
            const uint32_t c = draw_entry(a.tab, l, x.x, x.y);
            if (c) {
                pk[k] = l | (c << 16);
                atomicOr(&cb[k >> 5], 1u << (k & 31));
            }
        } else {
            pk[k] = 0;
        }
    }
    if (lane == 0) a.nnz_n[v] = nn;
    if (!do_draw) {
        for (int w = lane; w < KW; w += 32) nb[w] = 0;
        __syncwarp();
        return;
    }
    __syncwarp();
    // entries with n = 0: Pois(beta) by geometric skip-ahead (see phi_word)
    int pos = -1;
    for (uint32_t h0 = 0;; h0 += 32) {
        const U4 x = draw(a.seed, static_cast<uint32_t>(v), h0 + lane, sweep, TAG_BETA, 0);
        const int g = geo_gap(geo, x.x);
        const int step = g < 0 ? kGeoLen : g + 1;
        int incl = step;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
        }
        const int p = pos + incl;
        const bool stop = g < 0 ? p >= K - 1 : p >= K;
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, stop);
        const int first_stop = bal ? __ffs(bal) - 1 : 32;
        if (lane < first_stop && g >= 0 && pk[p] == 0) {
            const uint32_t c = table_draw(a.tab, 0, x.y, x.z);
            if (c) {
                pk[p] = c << 16;
                atomicOr(&cb[p >> 5], 1u << (p & 31));
            }
        }
        if (bal) break;
        pos = __shfl_sync(0xFFFFFFFFu, p, 31);
    }
    __syncwarp();
    // entries of n without a draw are cleared off the list of n, then the c column
    for (int i = lane; i < nn; i += 32) {
        const int k = list[i];
        if (pk[k] < 0x10000u) pk[k] = 0;
    }
    __syncwarp();
    const int nc = list_topics(cb, KW, list);
    for (int i = lane; i < nc; i += 32) {
        const int k = list[i];
        const uint32_t c = pk[k] >> 16;
        const int64_t o = static_cast<int64_t>(v) * K + i;
        pk[k] = 0;
        a.cst_k[o] = static_cast<uint16_t>(k);
        a.cst_c[o] = c;
        atomicAdd(&a.S[k], static_cast<u64>(c));
    }
    for (int w = lane; w < KW; w += 32) nb[w] = cb[w] = 0;
    if (lane == 0) a.nnz_c[v] = nc;
    __syncwarp();
}

// Shared memory of the count pass: a CTA's two K-entry arrays, or its warps'.
__host__ __device__ __forceinline__ int phi_count_words(int K) {
    const int w = K <= kWarpWordMaxK ? (kPhiCountBlock / 32) * warp_word_words(K) : 0;
    return w > 2 * K ? w : 2 * K;
}

// One chain's words, dynamically scheduled, most frequent first: the first
// n_big by the CTA (kPhiCountBlock threads: more words in flight per SM than
// with 256; a word's barriers then wait on fewer warps), the others by a warp
// each, kWarpWordBatch at a time.
constexpr int kWarpWordBatch = 4;
__global__ void __launch_bounds__(kPhiCountBlock) k_phi_counts(PhiArgs a, bool do_draw, int n_big) {
    extern __shared__ __align__(16) uint32_t sm[];
    __shared__ int scan_tmp[kPhiCountBlock / 32 + 1];
    __shared__ int s_item;
    __shared__ uint32_t geo[kGeoLen];
    for (int i = threadIdx.x; i < kGeoLen; i += kPhiCountBlock) geo[i] = a.tab.geo[i];
    if (threadIdx.x == 0) s_item = atomicAdd(a.work, 1);
    __syncthreads();
    for (;;) {
        const int item = s_item;      // published by the barrier above, then by phi_word's last one
        if (item >= n_big) break;
        phi_word<kPhiCountBlock>(a, a.word_order[item], do_draw, sm, sm + a.K, scan_tmp, geo, &s_item, a.work);
    }
    if (n_big >= a.V) return;
    const int lane = threadIdx.x & 31;
    uint32_t *pk = sm + static_cast<size_t>(threadIdx.x >> 5) * warp_word_words(a.K);
    __syncthreads();
    for (int i = lane; i < warp_word_words(a.K); i += 32) pk[i] = 0;
    __syncwarp();
    for (;;) {
        int first = 0;
        if (lane == 0) first = n_big + atomicAdd(a.work_warp, kWarpWordBatch);
        first = __shfl_sync(0xFFFFFFFFu, first, 0);
        if (first >= a.V) break;
        for (int i = first; i < min(first + kWarpWordBatch, a.V); ++i) phi_word_warp(a, a.word_order[i], do_draw, pk, a.K, geo);
    }
}

// Many chains: the work list holds (chain, word) pairs, most frequent first
// across all chains; shared memory is sized for the largest K.
__global__ void __launch_bounds__(kPhiCountBlock) k_phi_counts_multi(const PhiArgs *chains, const int2 *items, int n_items, int n_big,
                                                                 int *work, int *work_warp, int kmax, bool do_draw) {
    extern __shared__ __align__(16) uint32_t sm[];
    __shared__ int scan_tmp[kPhiCountBlock / 32 + 1];
    __shared__ int s_item;
    __shared__ uint32_t geo[kGeoLen];
    int geo_chain = -1;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(work, 1);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= n_big) break;
        const int2 it = items[item];
        if (it.x != geo_chain) {          // the geometric table depends on the chain's beta
            for (int i = threadIdx.x; i < kGeoLen; i += kPhiCountBlock) geo[i] = chains[it.x].tab.geo[i];
            geo_chain = it.x;
            __syncthreads();
        }
        phi_word<kPhiCountBlock>(chains[it.x], it.y, do_draw, sm, sm + kmax, scan_tmp, geo);
    }
    if (n_big >= n_items) return;
    const int lane = threadIdx.x & 31;
    uint32_t *pk = sm + static_cast<size_t>(threadIdx.x >> 5) * warp_word_words(kmax);
    for (int i = lane; i < warp_word_words(kmax); i += 32) pk[i] = 0;
    __syncwarp();
    for (;;) {
        int first = 0;
        if (lane == 0) first = n_big + atomicAdd(work_warp, kWarpWordBatch);
        first = __shfl_sync(0xFFFFFFFFu, first, 0);
        if (first >= n_items) break;
        for (int i = first; i < min(first + kWarpWordBatch, n_items); ++i) {
            const PhiArgs &a = chains[items[i].x];
            phi_word_warp(a, items[i].y, do_draw, pk, kmax, a.tab.geo);
        }
    }
}

// Topic histograms of the most frequent words, one chunk of a word's tokens
// per CTA, added into the word's row of heavy_hist (zero before: the count pass
// clears what it has read).
__device__ void heavy_chunk(const PhiArgs *chains, const HeavyChunk &c, uint32_t *hs) {
    const PhiArgs &a = chains[c.chain];
    const int K = a.K;
    for (int k = threadIdx.x; k < K; k += kPhiBlock) hs[k] = 0;
    __syncthreads();
    hist_tokens<kPhiBlock>(a, c.begin, c.end, hs);
    __syncthreads();
    uint32_t *row = a.heavy_hist + static_cast<int64_t>(c.row) * K;
    for (int k = threadIdx.x; k < K; k += kPhiBlock)
        if (hs[k]) atomicAdd(&row[k], hs[k]);
    __syncthreads();
}

__global__ void __launch_bounds__(kPhiBlock) k_heavy_hist(const PhiArgs *chains, const HeavyChunk *chunks) {
    extern __shared__ uint32_t hs[];
    heavy_chunk(chains, chunks[blockIdx.x], hs);
}

// n_{k,v} from the compacted n column of word v (binary search), 0 if absent.
__device__ uint32_t lookup_n(const PhiArgs &a, int v, int k) {
    const int64_t b = a.word_off[v];
    int lo = 0, hi = a.nnz_n[v];
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const int km = a.nst_k[b + mid];
        if (km < k) lo = mid + 1; else hi = mid;
    }
    return (lo < a.nnz_n[v] && a.nst_k[b + lo] == k) ? a.nst_n[b + lo] : 0u;
}

constexpr int kFixBlock = 1024;

// Rows whose Poisson counts summed to zero are redrawn whole (attempt
// a = 1, 2, ...) until the sum is nonzero: the urn total is Pois+ (the
// hierarchical representation, Eq. 8).  Accepted rows are inserted into the
// word columns.  One block of BLOCK threads; almost always just checks S and
// exits.  S is read from L2 (other CTAs of the same launch may have just
// summed it).
template <int BLOCK>
__device__ void phi_redraw_dead_rows(const PhiArgs &a, u64 *red, u64 *s_sum_p) {
    u64 &s_sum = *s_sum_p;
    const uint32_t sweep = sweep_of(a);
    // almost always no row is dead: one parallel look at S first
    int dead = 0;
    for (int k = threadIdx.x; k < a.K; k += BLOCK) dead |= __ldcg(&a.S[k]) == 0 ? 1 : 0;
    if (!__syncthreads_or(dead)) return;
    for (int k = 0; k < a.K; ++k) {
        if (__ldcg(&a.S[k]) != 0) continue;
        if (threadIdx.x == 0) atomicAdd(&a.stats[ST_DEADROWS], 1ull);
        uint32_t att = 1;
        for (; att <= kMaxRedraw; ++att) {
            u64 part = 0;
            for (int v = threadIdx.x; v < a.V; v += BLOCK) {
                const uint32_t l = lookup_n(a, v, k);
                uint32_t val = 0;
                if (l) {
                    const U4 x = draw(a.seed, static_cast<uint32_t>(v), static_cast<uint32_t>(k), sweep, TAG_REDRAW_POIS, att);
                    val = draw_entry(a.tab, l, x.x, x.y);
                }
                a.rowbuf[v] = val;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                int64_t pos = -1;
                uint32_t h = 0;
                for (;;) {
                    const U4 x = draw(a.seed, static_cast<uint32_t>(k), h++, sweep, TAG_REDRAW_BETA, att);
                    const int g = geo_gap(a.tab.geo, x.x);
                    if (g < 0) {
                        pos += kGeoLen;
                        if (pos >= a.V - 1) break;
                        continue;
                    }
                    pos += g + 1;
                    if (pos >= a.V) break;
                    if (lookup_n(a, static_cast<int>(pos), k) == 0) a.rowbuf[pos] = table_draw(a.tab, 0, x.y, x.z);
                }
            }
            __syncthreads();
            for (int v = threadIdx.x; v < a.V; v += BLOCK) part += a.rowbuf[v];
            part = warp_sum64(part);
            if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
            __syncthreads();
            if (threadIdx.x == 0) {
                u64 s = 0;
                for (int i = 0; i < BLOCK / 32; ++i) s += red[i];
                s_sum = s;
            }
            __syncthreads();
            const u64 sum = s_sum;
            if (sum > 0) {
                for (int v = threadIdx.x; v < a.V; v += BLOCK) {
                    const uint32_t val = a.rowbuf[v];
                    if (!val) continue;
                    const int64_t base = static_cast<int64_t>(v) * a.K;
                    int n = a.nnz_c[v];
                    int p = n;
                    while (p > 0 && a.cst_k[base + p - 1] > k) {
                        a.cst_k[base + p] = a.cst_k[base + p - 1];
                        a.cst_c[base + p] = a.cst_c[base + p - 1];
                        --p;
                    }
                    a.cst_k[base + p] = static_cast<uint16_t>(k);
                    a.cst_c[base + p] = val;
                    a.nnz_c[v] = n + 1;
                }
                if (threadIdx.x == 0) a.S[k] = sum;
                __syncthreads();
                break;
            }
            __syncthreads();
        }
        if (att > kMaxRedraw) {
            if (threadIdx.x == 0) atomicOr(&a.stats[ST_ERROR], ERR_DEGENERATE);
            return;
        }
    }
}

// The dead rows, then every row's reciprocal for the tables.
template <int BLOCK>
__device__ void phi_fixup_chain(const PhiArgs &a, u64 *red, u64 *s_sum_p) {
    phi_redraw_dead_rows<BLOCK>(a, red, s_sum_p);
    __syncthreads();
    for (int k = threadIdx.x; k < a.K; k += BLOCK) {
        const u64 S = __ldcg(&a.S[k]);
        a.rcp[k] = S ? static_cast<u64>(((static_cast<unsigned __int128>(1) << 127) - 1) / (S << __clzll(static_cast<long long>(S)))) : 0;
    }
}

__global__ void __launch_bounds__(kFixBlock) k_phi_fixup(PhiArgs a) {
    __shared__ u64 red[kFixBlock / 32];
    __shared__ u64 s_sum;
    phi_fixup_chain<kFixBlock>(a, red, &s_sum);
}

// Many chains: one CTA per chain.
__global__ void __launch_bounds__(kFixBlock) k_phi_fixup_multi(const PhiArgs *chains) {
    __shared__ u64 red[kFixBlock / 32];
    __shared__ u64 s_sum;
    phi_fixup_chain<kFixBlock>(chains[blockIdx.x], red, &s_sum);
}

// =================================================== Phi-step: tables
// Per word: phi = fp32(c/S) (Dirichlet mode: gamma (1/S), over the entries
// the selection kept); fixed-point weights q with
// 24 bits relative to the column maximum (q >= 1); alpha-part masses
// a = round(q alpha 2^16), A = sigma_a; Vose alias table over a; bitmap of
// the word's nonzero topics.
// One warp per word, the pairing included.  Vose's loop takes the small slots
// (mass below A) and the large ones each in descending slot order; a large
// slot whose mass falls below A is the next small one.  So the pairing is a
// merge of two running sums, the smalls' deficits D_i and the larges'
// excesses E_j:
//   small i goes to the first large j with E_j >= D_{i-1};
//   large j becomes small at the first i with D_i > E_j, with A + E_j - D_i
//   left, and goes to large j + 1;
// which one warp scan and a binary search per slot give, in exact integers.
// (In one lane, a step's loads in turn, it took 0.45 us per slot, and the
// longest columns were the whole pass: 455 us with K = 1000, 39 us with
// K = 100.)
constexpr int kTabSlots = 256;                                     // columns up to this long pair in shared memory
constexpr int kTabScratch = kTabSlots * (8 + 2);                   // bytes per warp
static_assert(kTabSlots * 8 >= 16384 / 8, "a word's bitmap is put together there too");

// The FP64 units are few (1.25 TFLOP/s), and some 45 FP64 instructions per
// entry bounded the pass (370 us for 100,000 words); the same values come
// from integers, with FP64 for one entry in 2^26.

// Mass of an entry of the alpha part: round(q alpha 2^16) in double, where
// every step is exact: q alpha has 49 bits, and so has the sum with 1/2.
__device__ __forceinline__ u64 alpha_mass(uint32_t q, float alpha) {
    const uint32_t b = __float_as_uint(alpha);
    const uint32_t ex = b >> 23;                              // alpha > 0
    const uint32_t ma = ex ? (b & 0x7FFFFFu) | 0x800000u : b;
    const int s = static_cast<int>(ex ? ex : 1) - 150 + 16;   // q alpha 2^16 = q ma 2^s
    const u64 x = static_cast<u64>(q) * ma;
    if (s >= 0) return x << s;
    return s > -64 ? (x + (1ull << (-s - 1))) >> -s : 0;
}

// p = c / S as (u / 2^63) 2^x, u in [2^62, 2^64) up to 3 below the exact value,
// and the exponent e of p = f 2^e, f in [1/2, 1).
struct Ratio { int x, e; };
__device__ __forceinline__ Ratio ratio_exponent(uint32_t c, u64 S) {
    const int zc = __clz(static_cast<int>(c)) + 32, zs = __clzll(static_cast<long long>(S));
    const int x = zs - zc;
    return {x, x + ((static_cast<u64>(c) << zc) >= (S << zs) ? 1 : 0)};
}

// max(1, floor(RN(c / S) 2^(24 - e) + 1/2)), the double expression's value.
// Double rounding and u move the product by less than 2^12 units of u, so
// integers decide unless the fraction is that close to 1/2.
__device__ __forceinline__ uint32_t fixed_weight(uint32_t c, u64 S, u64 rcp, int e) {
    const int zc = __clz(static_cast<int>(c)) + 32, zs = __clzll(static_cast<long long>(S));
    const u64 u = __umul64hi(static_cast<u64>(c) << zc, rcp);
    const int t = 39 + e - (zs - zc);                         // at least 39
    if (t > 63) return 1u;                                    // below 2^(24 - 24)
    const u64 half = 1ull << (t - 1), low = u & (2 * half - 1);
    u64 q = (u >> t) + (low >= half ? 1 : 0);
    if (low - half + 4096 < 8192) {
        const double scale = __longlong_as_double(static_cast<long long>(1023 + 24 - e) << 52);
        const double p = __ddiv_rn(static_cast<double>(c), static_cast<double>(S));
        q = static_cast<u64>(floor(__dadd_rn(__dmul_rn(p, scale), 0.5)));
    }
    return q < 1 ? 1u : static_cast<uint32_t>(q);
}

// The same for p given as a double > 0 (exact: p has 53 bits).
__device__ __forceinline__ uint32_t fixed_weight(long long pbits, int e) {
    const int ep = static_cast<int>(pbits >> 52);
    if (ep == 0) {                                            // subnormal p
        const double scale = __longlong_as_double(static_cast<long long>(1023 + 24 - e) << 52);
        const double q = floor(__dadd_rn(__dmul_rn(__longlong_as_double(pbits), scale), 0.5));
        return q < 1.0 ? 1u : static_cast<uint32_t>(q);
    }
    const u64 m = (static_cast<u64>(pbits) & ((1ull << 52) - 1)) | (1ull << 52);
    const int t = 1075 - ep - 24 + e;                         // p 2^(24 - e) = m 2^-t
    if (t > 62) return 1u;
    const u64 q = (m + (1ull << (t - 1))) >> t;
    return q < 1 ? 1u : static_cast<uint32_t>(q);
}

__device__ void phi_tables_word_warp(const PhiArgs &a, int v, uint8_t *stage, uint8_t *scratch) {
    const int lane = threadIdx.x & 31;
    const int n = a.nnz_c[v];
    const int64_t src = static_cast<int64_t>(v) * a.K;
    const int64_t out = a.col_ptr[v];
    if (a.bits) {
        // a row of KWp words (KW rounded up; the words past KW stay zero)
        uint32_t *bm = a.bits + static_cast<int64_t>(v) * a.KWp;
        uint32_t *sb = reinterpret_cast<uint32_t *>(scratch);
        for (int wi = lane; wi < a.KWp; wi += 32) sb[wi] = 0;
        __syncwarp();
        for (int j = lane; j < n; j += 32) {
            const int k = a.cst_k[src + j];
            atomicOr(&sb[k >> 5], 1u << (k & 31));
        }
        __syncwarp();
        for (int wi = lane; wi < a.KWp; wi += 32) bm[wi] = sb[wi];
        __syncwarp();
    }
    uint32_t *q32 = a.qdense ? a.qdense + static_cast<int64_t>(v) * a.K : nullptr;
    if (q32) {
        for (int k = lane; k < a.K; k += 32) q32[k] = 0;
        __syncwarp();
    }
    // the word's dense row is put together in `stage` (zero between words),
    // else in place
    const int slot = a.row_slot[v];
    const int RB = dense_row_bytes(a.K), PB = RB / 3;
    uint8_t *row = slot >= 0 ? a.qrow + static_cast<int64_t>(slot) * RB : nullptr;
    if (row && (n == 0 || !stage)) {
        for (int i = lane; i < RB / 16; i += 32) reinterpret_cast<uint4 *>(row)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
    }
    uint8_t *rw = stage ? stage : row;
    if (n == 0 && lane == 0) a.drow[v] = slot;
    if (n == 0) {
        if (lane == 0) a.A[v] = 0;
        return;
    }
    // the column's phi, then the running sums of the pairing; the slots by rank
    u64 *X = n <= kTabSlots ? reinterpret_cast<u64 *>(scratch) : a.vose_p + out;
    uint16_t *stk = n <= kTabSlots ? reinterpret_cast<uint16_t *>(scratch + 8 * kTabSlots) : a.vose_stack + out;
    // the column's largest phi is f 2^e, f in [1/2, 1)
    int e = -100000;
    for (int j = lane; j < n; j += 32) {
        const int k = a.cst_k[src + j];
        if (a.gam) {
            // gamma (1 / S_k), gamma's float bits staged in cst_c
            const long long p = __double_as_longlong(__dmul_rn(static_cast<double>(__uint_as_float(a.cst_c[src + j])), a.invS[k]));
            X[j] = static_cast<u64>(p);
            e = max(e, static_cast<int>(p >> 52) - 1022);
        } else {
            e = max(e, ratio_exponent(a.cst_c[src + j], __ldcg(&a.S[k])).e);
        }
    }
    e = __reduce_max_sync(0xFFFFFFFFu, e);
    u64 asum = 0;
    uint32_t qtop = 0;                  // a q of 2^24 does not fit a row's three bytes
    for (int j = lane; j < n; j += 32) {
        const int k = a.cst_k[src + j];
        const uint32_t c = a.cst_c[src + j];
        const uint32_t qv = a.gam ? fixed_weight(static_cast<long long>(X[j]), e) : fixed_weight(c, __ldcg(&a.S[k]), a.rcp[k], e);
        const u64 am = alpha_mass(qv, a.alpha[k]);
        a.topic[out + j] = static_cast<uint16_t>(k);
        a.c[out + j] = c;
        a.q[out + j] = qv;
        if (q32) q32[k] = qv;
        if (row) {
            const int at = dense_pos(a.K, k);
            rw[at] = static_cast<uint8_t>(qv);
            rw[at + PB] = static_cast<uint8_t>(qv >> 8);
            rw[at + 2 * PB] = static_cast<uint8_t>(qv >> 16);
        }
        qtop |= qv >> 24;
        asum += am;
    }
    asum = warp_sum64(asum);
    const bool fits = !__any_sync(0xFFFFFFFFu, qtop != 0);
    if (lane == 0) {
        a.A[v] = asum;
        a.drow[v] = fits ? slot : -1;
    }
    __syncwarp();
    if (row && stage) {
        for (int i = lane; i < RB / 16; i += 32) {
            reinterpret_cast<uint4 *>(row)[i] = reinterpret_cast<uint4 *>(stage)[i];
            reinterpret_cast<uint4 *>(stage)[i] = make_uint4(0u, 0u, 0u, 0u);
        }
        __syncwarp();
    }
    // Thresholds floor(P 2^32 / A) divide by the word's invariant A:
    // Moller and Granlund's 2/1 division with a reciprocal of the normalised
    // divisor, one 128-bit division per word instead of one per slot (exact).
    const int sh = asum ? __clzll(static_cast<long long>(asum)) : 0;
    const u64 dn = asum << sh;
    const u64 vinv = asum ? static_cast<u64>((~static_cast<unsigned __int128>(0)) / dn) : 0;   // floor((2^128-1)/dn) - 2^64
    auto store = [&](int j, int k, bool paired, int alias, u64 ps) {       // a slot that is not paired keeps its own topic
        u64 q1 = 0xFFFFFFFFu;
        if (paired) {
            // (u1, u0) = ps 2^32 2^sh, u1 < dn since ps < asum
            const u64 hi = ps >> 32, lo = ps << 32;
            const u64 u1 = sh ? (hi << sh) | (lo >> (64 - sh)) : hi;
            const u64 u0 = lo << sh;
            u64 q0 = vinv * u1;
            q1 = __umul64hi(vinv, u1);
            const u64 t = q0 + u0;
            q1 += u1 + (t < q0 ? 1ull : 0ull);
            q0 = t;
            q1 += 1;
            u64 r = u0 - q1 * dn;
            if (r > q0) { q1 -= 1; r += dn; }
            if (r >= dn) q1 += 1;
        }
        a.athr[out + j] = static_cast<uint32_t>(q1);
        a.atopic[out + j] = static_cast<uint16_t>(alias);
        if (a.apack) a.apack[out + j] = make_uint2(static_cast<uint32_t>(q1), static_cast<uint32_t>(k) | (static_cast<uint32_t>(alias) << 16));
    };
    const uint16_t *topic = a.topic + out;
    if (asum == 0) {
        for (int j = lane; j < n; j += 32) store(j, topic[j], false, topic[j], 0);
        return;
    }
    const u64 un = static_cast<u64>(n);                      // masses are scaled by n, so each slot holds A units
    if (__umul64hi(un, asum) == 0) {
        // X, stk: smalls from 0 up, larges from n - 1 down
        int ns = 0, nl = 0;
        u64 D = 0, E = 0;
        for (int j0 = 0; j0 < n; j0 += 32) {
            const int j = n - 1 - j0 - lane;
            const bool in = j >= 0;
            const u64 P = in ? alpha_mass(a.q[out + j], a.alpha[topic[j]]) * un : 0;
            const bool small = in && P < asum, large = in && !small;
            const uint32_t bs = __ballot_sync(0xFFFFFFFFu, small), bl = __ballot_sync(0xFFFFFFFFu, large);
            const uint32_t below = (1u << lane) - 1u;
            const u64 d = D + warp_incl_scan(small ? asum - P : 0), e = E + warp_incl_scan(large ? P - asum : 0);
            if (in) {
                const int at = small ? ns + __popc(bs & below) : n - 1 - (nl + __popc(bl & below));
                X[at] = small ? d : e;
                stk[at] = static_cast<uint16_t>(j);
            }
            D = __shfl_sync(0xFFFFFFFFu, d, 31);
            E = __shfl_sync(0xFFFFFFFFu, e, 31);
            ns += __popc(bs);
            nl += __popc(bl);
        }
        __syncwarp();
        for (int i = lane; i < n; i += 32) {
            const int j = stk[i], k = topic[j];
            const u64 x = X[i];
            bool paired;
            int to = i;                                      // whose topic is the alias
            u64 ps = 0;
            if (i < ns) {
                const u64 before = i ? X[i - 1] : 0;
                int lo = 0, hi = nl;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (X[n - 1 - mid] < before) lo = mid + 1; else hi = mid;
                }
                paired = lo < nl;
                if (paired) { to = n - 1 - lo; ps = asum - (x - before); }
            } else {
                int lo = 0, hi = ns;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (X[mid] <= x) lo = mid + 1; else hi = mid;
                }
                paired = lo < ns && i > ns;                  // a next large one exists
                if (paired) { to = i - 1; ps = asum + x - X[lo]; }
            }
            store(j, k, paired, topic[stk[to]], ps);
        }
        __syncwarp();
        return;
    }
    // the sums do not fit 64 bits (long columns with large alpha): Vose's loop in lane 0
    u64 *P = a.vose_p + out;
    uint16_t *st = a.vose_stack + out;
    int ns = 0, nl = 0;
    for (int j0 = 0; j0 < n; j0 += 32) {
        const int j = j0 + lane;
        const bool in = j < n;
        const u64 p = in ? alpha_mass(a.q[out + j], a.alpha[topic[j]]) * un : 0;
        const bool small = in && p < asum;
        const uint32_t bs = __ballot_sync(0xFFFFFFFFu, small), bl = __ballot_sync(0xFFFFFFFFu, in && !small);
        const uint32_t below = (1u << lane) - 1u;
        if (in) {
            P[j] = p;
            a.atopic[out + j] = topic[j];
            st[small ? ns + __popc(bs & below) : n - 1 - (nl + __popc(bl & below))] = static_cast<uint16_t>(j);
        }
        ns += __popc(bs);
        nl += __popc(bl);
    }
    __syncwarp();
    if (lane == 0) {
        while (ns > 0 && nl > 0) {
            const int s = st[--ns];
            --nl;
            const int l = st[n - 1 - nl];
            const u64 ps = P[s];             // final: s is not pushed again
            a.atopic[out + s] = topic[l];
            const u64 pl = P[l] - (asum - ps);
            P[l] = pl;
            if (pl < asum) st[ns++] = static_cast<uint16_t>(l);
            else { st[n - 1 - nl] = static_cast<uint16_t>(l); ++nl; }
        }
    }
    __syncwarp();
    for (int j = lane; j < n; j += 32) store(j, topic[j], a.atopic[out + j] != topic[j], a.atopic[out + j], P[j]);
    __syncwarp();
}

// A warp's part of the shared memory: kTabScratch bytes, and where the CTA has
// the room the stage of the dense row it puts together (stage_bytes, zeroed;
// else null).
struct TableMem { uint8_t *stage, *scratch; };
__device__ __forceinline__ TableMem table_mem(uint32_t *sm, int stage_bytes) {
    uint8_t *base = reinterpret_cast<uint8_t *>(sm) + static_cast<size_t>(threadIdx.x >> 5) * (stage_bytes + kTabScratch);
    TableMem t{stage_bytes ? base + kTabScratch : nullptr, base};
    for (int i = threadIdx.x & 31; i < stage_bytes / 16; i += 32) reinterpret_cast<uint4 *>(t.stage)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    return t;
}

// One warp per word, most frequent first (their columns are the longest).
__global__ void k_phi_tables(PhiArgs a, int stage_bytes) {
    extern __shared__ __align__(16) uint32_t tsm[];
    const TableMem t = table_mem(tsm, stage_bytes);
    const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = wid; i < a.V; i += nwarps) phi_tables_word_warp(a, a.word_order[i], t.stage, t.scratch);
}

__global__ void k_phi_tables_multi(const PhiArgs *chains, const int2 *items, int n_items, int stage_bytes) {
    extern __shared__ __align__(16) uint32_t tsm[];
    const TableMem t = table_mem(tsm, stage_bytes);
    const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = wid; i < n_items; i += nwarps) {
        const int2 it = items[i];
        phi_tables_word_warp(chains[it.x], it.y, t.stage, t.scratch);
    }
}

// ============================================================== z-step
// 4-warp CTAs, 7 per SM: 72 registers, 28 warps per SM.
#ifndef PULDA_ZMINBLOCKS
#define PULDA_ZMINBLOCKS 7
#endif

// One chain, one document per warp (dynamically scheduled, longest first),
// one pass.
// NW = z_nw(K) words per lane and plane, one instantiation per kernel.
template <int NW>
__global__ void __launch_bounds__(32 * kZWarps, NW < 0 ? 2 : PULDA_ZMINBLOCKS) k_z_step(ZArgs a) {
    extern __shared__ __align__(16) uint32_t zsm[];
    const int lane = threadIdx.x & 31;
    uint32_t *m = zsm + static_cast<size_t>(threadIdx.x >> 5) * z_dense_warp_words(a.K, a.narrow != 0);
    u64 *wcnt = z_dense_counters(m, a.K, a.narrow != 0);
    zero_warp_counters(wcnt);
    const uint32_t sweep = sweep_of(a);
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(a.work, 1);
        item = __shfl_sync(0xFFFFFFFFu, item, 0);
        if (item >= a.n_slices + a.D) break;
        int64_t s;
        int len;
        const uint32_t *m0 = nullptr;
        if (item < a.n_slices) {
            // a slice of a long document: {document, its row in m0, first token, tokens}
            const int4 sl = a.slices[item];
            s = a.doc_off[sl.x] + sl.z;
            len = sl.w;
            m0 = a.m0 + static_cast<int64_t>(sl.y) * a.K;
        } else {
            const int d = a.doc_order[item - a.n_slices];
            s = a.doc_off[d];
            len = static_cast<int>(a.doc_off[d + 1] - s);
        }
        DocRun r{a.w + s, a.z + s, len, a.seed, a.index_base + s, sweep, 0, len, 1};
        z_doc<NW>(a, m, r, wcnt, m0);
    }
    flush_warp_counters(a.stats, wcnt);
}

#ifndef PULDA_PAIR_MINB
#define PULDA_PAIR_MINB 8
#endif
// The same with two documents per warp, of at most kNarrowMaxLen tokens each
// (neighbours of the length order, so their lengths are near); no slices.
template <int NW>
__global__ void __launch_bounds__(32 * kZWarps, PULDA_PAIR_MINB) k_z_step_pairs(ZArgs a) {
    extern __shared__ __align__(16) uint32_t zsm[];
    const int lane = threadIdx.x & 31;
    uint32_t *m = zsm + static_cast<size_t>(threadIdx.x >> 5) * z_pair_words(a.K);
    u64 *wcnt = reinterpret_cast<u64 *>(m + 2 * 2 * 32 * NW + 32 * kTokRecWords);
    zero_warp_counters(wcnt);
    const uint32_t sweep = sweep_of(a);
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(a.work, 1);
        item = __shfl_sync(0xFFFFFFFFu, item, 0);
        if (2 * static_cast<int64_t>(item) >= a.D) break;
        const int64_t di = 2 * static_cast<int64_t>(item) + (lane >> 4);
        int64_t s = 0;
        int len = 0;
        if (di < a.D) {
            const int d = a.doc_order[di];
            s = a.doc_off[d];
            len = static_cast<int>(a.doc_off[d + 1] - s);
        }
        const DocRun r{a.w + s, a.z + s, len, a.seed, a.index_base + s, sweep, 0, len, 1};
        z_pair<NW>(a, m, r, wcnt);
    }
    flush_warp_counters(a.stats, wcnt);
}

// m0[j * K + k] = the topic-k count of document sliced_docs[j] (one warp per
// document): the pass-start counts its slices start from.
__global__ void k_slice_counts(const int64_t *doc_off, const int32_t *sliced_docs, int n, const int16_t *z, int K,
                               uint32_t *m0) {
    const int lane = threadIdx.x & 31;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < n; j += nwarps) {
        uint32_t *row = m0 + static_cast<int64_t>(j) * K;
        for (int k = lane; k < K; k += 32) row[k] = 0;
        __syncwarp();
        const int d = sliced_docs[j];
        for (int64_t i = doc_off[d] + lane; i < doc_off[d + 1]; i += 32) atomicAdd(&row[z[i]], 1u);
        __syncwarp();
    }
}

// Many chains of one form (NW): items[0 .. n_items) are (chain, document)
// pairs, longest first, taken one after another by every warp.  m: the warp's
// area, sized for kmax topics.
template <int NW>
__device__ __forceinline__ void z_multi_items(const ZArgs *chains, const int2 *items, int n_items, int *work, uint32_t *m, u64 *wcnt,
                                              int narrow) {
    const int lane = threadIdx.x & 31;
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(work, 1);
        item = __shfl_sync(0xFFFFFFFFu, item, 0);
        if (item >= n_items) break;
        const int2 it = items[item];
        ZArgs a = chains[it.x];         // a copy: the token loop's stores would have its fields read again
        a.narrow = narrow;
        const int64_t s = a.doc_off[it.y];
        const int len = static_cast<int>(a.doc_off[it.y + 1] - s);
        DocRun r{a.w + s, a.z + s, len, a.seed, a.index_base + s, sweep_of(a), 0, len, 1};
        z_doc<NW>(a, m, r, wcnt, nullptr);
        flush_warp_counters(a.stats, wcnt);
    }
}

template <int NW>
__global__ void __launch_bounds__(32 * kMultiWarps, PULDA_MULTI_MINB) k_z_step_multi(const ZArgs *chains, const int2 *items,
                                                                        int n_items, int *work, int kmax, int narrow) {
    extern __shared__ __align__(16) uint32_t zsm[];
    uint32_t *m = zsm + static_cast<size_t>(threadIdx.x >> 5) * z_dense_warp_words(kmax, narrow != 0);
    u64 *wcnt = z_dense_counters(m, kmax, narrow != 0);     // beyond every chain's counts and token records
    zero_warp_counters(wcnt);
    z_multi_items<NW>(chains, items, n_items, work, m, wcnt, narrow);
}

// ============================================================ batches
// Start of a sweep of many chains (one CTA): advance the shared sweep counter
// and clear every chain's row sums, per-sweep counters and the work queues.
__device__ void batch_begin_sweep(const PhiArgs *chains, int n_chains, uint32_t *sweep, int *work) {
    if (threadIdx.x == 0) *sweep += 1u;
    if (threadIdx.x < kBatchCounters) work[threadIdx.x] = 0;
    for (int c = 0; c < n_chains; ++c) {
        const PhiArgs &a = chains[c];
        for (int k = threadIdx.x; k < a.K; k += blockDim.x) a.S[k] = 0;
        for (int i = threadIdx.x; i < ST_COUNT; i += blockDim.x) a.stats[i] = 0;
    }
}

__global__ void k_batch_begin_sweep(const PhiArgs *chains, int n_chains, uint32_t *sweep, int *work) {
    batch_begin_sweep(chains, n_chains, sweep, work);
}

// ============================================================ serving
// One step of the fold-in server: each active slot (a request's document,
// resampled with Phi fixed) advances by up to `slice` tokens, continuing
// across passes, one warp per slot.  A slot whose pass counter is 0 first
// gets its uniform initial topics (counter 0, as pulda_infer).  The slot's
// (pass, position) is written back for the host's completion check.
// Its slot bookkeeping needs a few more registers than k_z_step: 7 CTAs per
// SM keep it free of spills.
// With window_ns > 0 a slot also stops at the first 32-token block boundary
// window_ns after its warp took it up, having done at least one block (a slot
// taken up in a later wave of a crowded launch gets the same time as the first).
template <int NW>
__global__ void __launch_bounds__(32 * kZWarps, 7) k_serve_step(ZArgs a, ServeSlot *slots, const int32_t *active,
                                                                     int n_active, const int32_t *arena_w,
                                                                     int16_t *arena_z, int64_t slice, int *work,
                                                                     uint64_t window_ns) {
    extern __shared__ __align__(16) uint32_t zsm[];
    const int lane = threadIdx.x & 31;
    uint32_t *m = zsm + static_cast<size_t>(threadIdx.x >> 5) * z_dense_warp_words(a.K, a.narrow != 0);
    u64 *wcnt = z_dense_counters(m, a.K, a.narrow != 0);
    zero_warp_counters(wcnt);
    for (;;) {
        int item = 0;
        uint64_t t0 = 0;
        if (lane == 0) {
            item = atomicAdd(work, 1);
            if (window_ns) t0 = global_ns();
        }
        item = __shfl_sync(0xFFFFFFFFu, item, 0);
        if (item >= n_active) break;
        const uint64_t deadline = window_ns ? __shfl_sync(0xFFFFFFFFu, t0, 0) + window_ns : ~0ull;
        const int idx = active[item];
        const ServeSlot sl = slots[idx];
        int16_t *z = arena_z + sl.off;
        uint32_t sweep = sl.sweep;
        int pos = sl.pos;
        if (sweep == 0) {
            for (int i = lane; i < sl.len; i += 32) {
                const U4 x = draw(sl.seed, static_cast<uint32_t>(i), 0u, 0u, TAG_INIT, 0);
                z[i] = static_cast<int16_t>(__umulhi(x.x, static_cast<uint32_t>(a.K)));
            }
            __syncwarp();
            sweep = 1;
            pos = 0;
        }
        DocRun r{arena_w + sl.off, z, sl.len, sl.seed, 0, sweep, pos, slice,
                 static_cast<int>(sl.sweep_end - sweep), deadline};
        z_doc<NW>(a, m, r, wcnt, nullptr);
        if (lane == 0) {
            slots[idx].sweep = r.sweep;
            slots[idx].pos = r.pos;
        }
    }
    flush_warp_counters(a.stats, wcnt);
}

// ============================================================== exports
// m_{d,k}, dense row-major [D, K]: one warp per document.
__global__ void k_doc_topic(const int64_t *doc_off, int64_t D, const int16_t *z, int K, int32_t *m_dk) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
    const int64_t nw = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    for (int64_t d = gw; d < D; d += nw) {
        int32_t *row = m_dk + d * K;
        for (int64_t i = doc_off[d] + lane; i < doc_off[d + 1]; i += 32) atomicAdd(&row[z[i]], 1);
    }
}

// n_{k,v}, dense row-major [K, V], from the compacted n columns.
__global__ void k_n_dense(PhiArgs a, int32_t *n_kv) {
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < a.V; v += gridDim.x * blockDim.x) {
        const int64_t b = a.word_off[v];
        for (int j = 0; j < a.nnz_n[v]; ++j) n_kv[static_cast<int64_t>(a.nst_k[b + j]) * a.V + v] = static_cast<int32_t>(a.nst_n[b + j]);
    }
}

// phi_{k,v} = fp32(c_{k,v} / S_k) for every stored entry (Dirichlet mode:
// fp32(gamma_{k,v} (1 / S_k))).
__global__ void k_phi_values(PhiArgs a, float *phi) {
    const int64_t nnz = a.col_ptr[a.V];
    for (int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; e < nnz;
         e += static_cast<int64_t>(gridDim.x) * blockDim.x)
        phi[e] = a.gam ? static_cast<float>(__dmul_rn(static_cast<double>(__uint_as_float(a.c[e])), a.invS[a.topic[e]]))
                       : static_cast<float>(__ddiv_rn(static_cast<double>(a.c[e]), static_cast<double>(a.S[a.topic[e]])));
}

int sm_count() {
    static int n = 0;
    if (!n) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
    }
    return n;
}

}  // namespace

// ============================================================ launchers
void launch_init_z(int64_t N, int K, uint64_t seed, int64_t index_base, int16_t *z, cudaStream_t st) {
    if (N <= 0) return;
    const int grid = static_cast<int>(std::min<int64_t>((N + 255) / 256, 8LL * sm_count() * 8));
    k_init_z<<<grid, 256, 0, st>>>(N, K, seed, index_base, z);
}

void launch_word_perm(int64_t N, int V, const int32_t *w, int64_t *word_off, int32_t *fill, int32_t *perm,
                      cudaStream_t st) {
    cudaMemsetAsync(fill, 0, sizeof(int32_t) * V, st);
    const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((N + 255) / 256, 8LL * sm_count() * 8)));
    if (N > 0) k_word_hist<<<grid, 256, 0, st>>>(N, w, fill);
    k_scan<<<scan_chunks(V), kScanBlock, 0, st>>>(fill, V, word_off, nullptr);
    cudaMemsetAsync(fill, 0, sizeof(int32_t) * V, st);
    if (N > 0) k_word_scatter<<<grid, 256, 0, st>>>(N, w, word_off, fill, perm);
}

size_t phi_counts_smem(int K) { return sizeof(uint32_t) * 2 * static_cast<size_t>(K); }

// The words that a CTA counts each, of n of which n_over have more than
// phi_warp_word_tokens() tokens: those, or all where a warp's counts do not fit
// or one wave of the grid's CTAs has them all (a warp takes longer over a word,
// and nothing waits for the CTA then).
int phi_big_words(int K, int64_t n, int64_t n_over, int grid) {
    return static_cast<int>(K <= kWarpWordMaxK && n > grid ? n_over : n);
}
int64_t phi_warp_word_tokens() { return kWarpWord; }

// The dynamic shared-memory opt-in is a per-kernel attribute shared by every
// handle in the process, so it is set once to the device maximum.
int smem_optin() {
    static int v = 0;
    if (!v) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (v <= 0) v = 48 * 1024;
    }
    return v;
}

int phi_counts_blocks_per_sm(int K) {
    const size_t smem = sizeof(uint32_t) * phi_count_words(K);
    allow_dynamic_smem(k_phi_counts);
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_phi_counts, kPhiCountBlock, smem);
    return b > 0 ? b : 1;
}

void launch_phi_counts(const PhiArgs &a, bool draw, int grid, cudaStream_t st) {
    // columns built by the sort path are the CTA's to read
    const int n_big = a.counted ? a.V : std::min(a.n_big, a.V);
    k_phi_counts<<<grid, kPhiCountBlock, sizeof(uint32_t) * phi_count_words(a.K), st>>>(a, draw, n_big);
}

void launch_phi_fixup(const PhiArgs &a, cudaStream_t st) { k_phi_fixup<<<1, kFixBlock, 0, st>>>(a); }

void launch_colptr_scan(const PhiArgs &a, cudaStream_t st) {
    k_scan<<<scan_chunks(a.V), kScanBlock, 0, st>>>(a.nnz_c, a.V, a.col_ptr, &a.stats[ST_NNZPHI]);
}

// Warps per CTA and stage bytes per warp of the table pass: eight warps while
// their stages stay within 96 KB, fewer for the longest rows.
static int table_warps(int K) {
    int w = 8;
    while (w > 1 && w * dense_row_bytes(K) > 96 * 1024) w >>= 1;
    return w;
}

static std::atomic<bool> g_tables_opted{false};
static void opt_in_tables() {
    if (g_tables_opted.load(std::memory_order_acquire)) return;
    allow_dynamic_smem(k_phi_tables);
    allow_dynamic_smem(k_phi_tables_multi);
    g_tables_opted.store(true, std::memory_order_release);
}

void launch_phi_tables(const PhiArgs &a, cudaStream_t st) {
    opt_in_tables();
    const int w = table_warps(a.K), rb = dense_row_bytes(a.K);
    const int grid = static_cast<int>(std::min<int64_t>((a.V + w - 1) / w, 128LL / w * sm_count()));
    k_phi_tables<<<std::max(grid, 1), 32 * w, static_cast<size_t>(w) * (rb + kTabScratch), st>>>(a, rb);
}

void launch_phi_tables_multi(const PhiArgs *chains, const int2 *items, int n_items, int kmax, cudaStream_t st) {
    opt_in_tables();
    const int w = table_warps(kmax), rb = dense_row_bytes(kmax);
    const int grid = static_cast<int>(std::min<int64_t>((n_items + w - 1) / w, 128LL / w * sm_count()));
    k_phi_tables_multi<<<std::max(grid, 1), 32 * w, static_cast<size_t>(w) * (rb + kTabScratch), st>>>(chains, items, n_items, rb);
}

void launch_heavy_hist(const PhiArgs *chains, const HeavyChunk *chunks, int n_chunks, int kmax, cudaStream_t st) {
    if (n_chunks <= 0) return;
    static bool opted_in = false;
    if (!opted_in) { allow_dynamic_smem(k_heavy_hist); opted_in = true; }
    k_heavy_hist<<<n_chunks, kPhiBlock, sizeof(uint32_t) * static_cast<size_t>(kmax), st>>>(chains, chunks);
}

size_t z_step_smem(int K, int warps_per_block, bool narrow) {
    return sizeof(uint32_t) * static_cast<size_t>(z_dense_warp_words(K, narrow)) * warps_per_block;
}

using ZStepKernel = void (*)(ZArgs);
static ZStepKernel z_step_kernel(int K) {
    switch (z_nw(K)) {
        case 1: return k_z_step<1>;
        case 2: return k_z_step<2>;
        case 4: return k_z_step<4>;
        case 8: return k_z_step<8>;
        default: return k_z_step<0>;
    }
}

static ZStepKernel z_pair_kernel(int K) {
    switch (z_nw(K)) {
        case 1: return k_z_step_pairs<1>;
        case 2: return k_z_step_pairs<2>;
        case 4: return k_z_step_pairs<4>;
        case 8: return k_z_step_pairs<8>;
        default: return nullptr;
    }
}

int z_pair_blocks_per_sm(int K, int warps_per_block) {
    ZStepKernel kern = z_pair_kernel(K);
    if (!kern) return 0;
    allow_dynamic_smem(kern);
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, 32 * warps_per_block, sizeof(uint32_t) * z_pair_words(K) * warps_per_block);
    return b;
}

void launch_z_step_pairs(const ZArgs &a, int warps_per_block, int grid, cudaStream_t st) {
    z_pair_kernel(a.K)<<<grid, 32 * warps_per_block, sizeof(uint32_t) * z_pair_words(a.K) * warps_per_block, st>>>(a);
}

int z_step_blocks_per_sm(int K, int warps_per_block, bool narrow) {
    const size_t smem = z_step_smem(K, warps_per_block, narrow);
    ZStepKernel kern = z_step_kernel(K);
    allow_dynamic_smem(kern);
    if (z_nw(K) == 0) allow_dynamic_smem(k_z_step<-1>);      // for launch_z_step, which loads no kernel
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, 32 * warps_per_block, smem);
    return b > 0 ? b : 1;
}

void launch_slice_counts(const int64_t *doc_off, const int32_t *sliced_docs, int n, const int16_t *z, int K,
                         uint32_t *m0, cudaStream_t st) {
    if (n <= 0) return;
    const int grid = std::max(1, std::min((n + 7) / 8, 4 * sm_count()));
    k_slice_counts<<<grid, 256, 0, st>>>(doc_off, sliced_docs, n, z, K, m0);
}

void launch_z_step(const ZArgs &a, int warps_per_block, int grid, cudaStream_t st) {
    // Few documents, each bound by its loads' latency, take the form that has more
    // of them in flight: above 1,024 topics where one has 2^16 tokens or more,
    // above 4,096 always (100 documents of 200 tokens, ms: K = 8,000 1.55 -> 1.15,
    // K = 16,384 4.4 -> 2.7; 700 beside documents on CTAs, whose SMs it shares
    // worse: K = 3,000 0.64 -> 0.80, K = 8,000 1.07 -> 0.86)
    const bool few = (a.K > 4096 || a.narrow == 0) && a.n_slices == 0 && a.D <= 4 * static_cast<int64_t>(sm_count()) && z_nw(a.K) == 0;
    const ZStepKernel kern = few ? k_z_step<-1> : z_step_kernel(a.K);
    kern<<<grid, 32 * warps_per_block, z_step_smem(a.K, warps_per_block, a.narrow != 0), st>>>(a);
}

using ZMultiKernel = void (*)(const ZArgs *, const int2 *, int, int *, int, int);
static ZMultiKernel z_multi_kernel(int kmax) {
    switch (z_nw(kmax)) {
        case 1: return k_z_step_multi<1>;
        case 2: return k_z_step_multi<2>;
        case 4: return k_z_step_multi<4>;
        case 8: return k_z_step_multi<8>;
        default: return k_z_step_multi<0>;
    }
}

static void launch_z_step_multi(const BatchLaunch &b, const BatchForm &f, const int2 *items, int n, bool narrow, int *work,
                                cudaStream_t st) {
    if (n <= 0) return;
    const int grid = std::min(f.z_grid, (n + b.z_warps - 1) / b.z_warps);
    z_multi_kernel(f.kmax)<<<grid, 32 * b.z_warps, z_step_smem(f.kmax, b.z_warps, narrow), st>>>(b.z, items, n, work, f.kmax,
                                                                                                narrow ? 1 : 0);
}

// The chains' documents by form, the longest ones of each on CTAs beside the
// others: every launch on a stream of its own (the CTAs first), so that one's
// last documents do not hold up the next.
static void launch_batch_z(const BatchLaunch &b, cudaStream_t st) {
    cudaEventRecord(b.ev_fork, st);
    int used = 0;
    auto branch = [&](auto launch) {
        cudaStream_t s = used == 0 ? st : b.side[used - 1];
        if (used > 0) cudaStreamWaitEvent(s, b.ev_fork, 0);
        launch(s);
        ++used;
    };
    for (int f = 0; f < b.n_forms; ++f) {
        const BatchForm &F = b.form[f];
        const int2 *items = b.form_items + F.first;
        if (std::max(F.n_wide, F.n_coop) > 0)
            branch([&](cudaStream_t s) {
                launch_z_step_coop_multi(b.z, items, F.n_coop, F.n_wide > 0, b.work + 3 + 3 * f, F.kmax, F.coop_grid, s);
                launch_z_step_multi(b, F, items + F.n_coop, F.n_wide - F.n_coop, false, b.work + 2 + 3 * f, s);
            });
    }
    for (int f = 0; f < b.n_forms; ++f) {
        const BatchForm &F = b.form[f];
        const int head = std::max(F.n_wide, F.n_coop);
        if (F.n > head)
            branch([&](cudaStream_t s) {
                launch_z_step_multi(b, F, b.form_items + F.first + head, F.n - head, true, b.work + 4 + 3 * f, s);
            });
    }
    for (int i = 1; i < used; ++i) {
        cudaEventRecord(b.ev_join[i - 1], b.side[i - 1]);
        cudaStreamWaitEvent(st, b.ev_join[i - 1], 0);
    }
}

void launch_batch_sweep(const BatchLaunch &b, cudaStream_t st) {
    k_batch_begin_sweep<<<1, 256, 0, st>>>(b.phi, b.n_chains, b.sweep, b.work);
    launch_heavy_hist(b.phi, b.heavy, b.n_heavy, b.kmax, st);
    k_phi_counts_multi<<<b.phi_grid, kPhiCountBlock, sizeof(uint32_t) * phi_count_words(b.kmax), st>>>(
        b.phi, b.phi_items, b.n_phi_items, std::min(b.n_big, b.n_phi_items), b.work, b.work + 1, b.kmax, true);
    k_phi_fixup_multi<<<b.n_chains, kFixBlock, 0, st>>>(b.phi);
    k_colptr_scan_multi<<<dim3(b.n_chains, scan_chunks(b.vmax)), kScanBlock, 0, st>>>(b.phi);
    launch_phi_tables_multi(b.phi, b.phi_items, b.n_phi_items, b.kmax, st);
    launch_batch_z(b, st);
}

// ---------------------------------------------------------- one persistent launch per Phi-step
// The same Phi-step of many chains as launch_batch_sweep's, in one cooperative
// launch whose CTAs are all resident: the phases (counter reset, heavy-word
// histograms, counts and draws, dead-row redraws, column offsets, per-word
// tables) run one after another, each over the whole grid, separated by a grid
// barrier.  The z-step follows in its own launches: five forms of it in this
// kernel took 128 registers, so 16 warps per SM against their 28 (99.9M tokens
// in eight chains: a sweep took 46 ms).  Nothing a phase reads was read earlier in the launch by
// another SM before its writers finished (so no stale L1 line is read), except
// the row sums and heavy-word histograms, which are read from L2.
constexpr int kPersistThreads = 256;
constexpr int kPersistWarps = kPersistThreads / 32;
// A grid barrier with a bounded wait: thread 0 of each CTA arrives; the last
// to arrive opens the next generation.  A CTA that has waited 2 s sets
// ERR_BARRIER in err and returns false (the launch then ends with an error
// instead of waiting forever).
__device__ bool grid_barrier(GridBarrier *bar, unsigned nblocks, unsigned long long *err) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        s_ok = 1;
        volatile unsigned *gen = &bar->gen;
        const unsigned g = *gen;
        __threadfence();
        if (atomicAdd(&bar->count, 1u) == nblocks - 1) {
            atomicExch(&bar->count, 0u);
            __threadfence();
            atomicAdd(&bar->gen, 1u);
        } else {
            const uint64_t t0 = global_ns();
            while (*gen == g) {
                if (global_ns() - t0 > 2000000000ull) {
                    atomicOr(err, ERR_BARRIER);
                    s_ok = 0;
                    break;
                }
                __nanosleep(100);
            }
        }
        __threadfence();
    }
    __syncthreads();
    return s_ok != 0;
}

// The barrier alone, for its self-test: every CTA passes `rounds` barriers
// that expect `expect` arrivals.
__global__ void k_barrier_selftest(GridBarrier *bar, unsigned expect, int rounds, unsigned long long *err,
                                   unsigned *passed) {
    for (int r = 0; r < rounds; ++r) {
        if (!grid_barrier(bar, expect, err)) return;
        if (threadIdx.x == 0) atomicAdd(passed, 1u);
    }
}

__global__ void __launch_bounds__(kPersistThreads, 4) k_batch_sweep_persistent(BatchLaunch b) {
    extern __shared__ __align__(16) uint32_t psm[];
    __shared__ int scan_tmp[kPersistThreads / 32 + 1];
    __shared__ int s_item;
    __shared__ uint32_t geo[kGeoLen];
    __shared__ u64 red[kPersistThreads / 32];
    __shared__ u64 s_sum;
    const unsigned nb = gridDim.x;
    unsigned long long *err = b.phi[0].stats + ST_ERROR;
    // counters of the sweep
    if (blockIdx.x == 0) batch_begin_sweep(b.phi, b.n_chains, b.sweep, b.work);
    if (!grid_barrier(b.bar, nb, err)) return;
    // histograms of the most frequent words, chunk by chunk
    for (int c = blockIdx.x; c < b.n_heavy; c += nb) heavy_chunk(b.phi, b.heavy[c], psm);
    if (!grid_barrier(b.bar, nb, err)) return;
    // counts and Poisson draws, (chain, word) items most frequent first
    {
        int geo_chain = -1;
        for (;;) {
            if (threadIdx.x == 0) s_item = atomicAdd(&b.work[0], 1);
            __syncthreads();
            const int item = s_item;
            __syncthreads();
            if (item >= b.n_phi_items) break;
            const int2 it = b.phi_items[item];
            if (it.x != geo_chain) {
                for (int i = threadIdx.x; i < kGeoLen; i += kPersistThreads) geo[i] = b.phi[it.x].tab.geo[i];
                geo_chain = it.x;
                __syncthreads();
            }
            phi_word<kPersistThreads>(b.phi[it.x], it.y, true, psm, psm + b.kmax, scan_tmp, geo);
        }
    }
    if (!grid_barrier(b.bar, nb, err)) return;
    // rows whose draws summed to zero, one CTA per chain
    for (int c = blockIdx.x; c < b.n_chains; c += nb) phi_fixup_chain<kPersistThreads>(b.phi[c], red, &s_sum);
    if (!grid_barrier(b.bar, nb, err)) return;
    const int per_chain = scan_chunks(b.vmax);
    for (int c = blockIdx.x; c < b.n_chains * per_chain; c += nb) {
        const PhiArgs &a = b.phi[c / per_chain];
        if (c % per_chain < scan_chunks(a.V))
            scan_one_chunk<kPersistThreads>(a.nnz_c, a.V, a.col_ptr, &a.stats[ST_NNZPHI], c % per_chain, scan_tmp, red);
    }
    if (!grid_barrier(b.bar, nb, err)) return;
    // per-word tables, one warp per (chain, word)
    {
        const int wid = static_cast<int>(blockIdx.x) * kPersistWarps + (threadIdx.x >> 5);
        const int nw = static_cast<int>(nb) * kPersistWarps;
        const TableMem t = table_mem(psm, b.table_stage);
        for (int i = wid; i < b.n_phi_items; i += nw) {
            const int2 it = b.phi_items[i];
            phi_tables_word_warp(b.phi[it.x], it.y, t.stage, t.scratch);
        }
    }
}

cudaError_t launch_barrier_selftest(GridBarrier *bar, int blocks, int missing, int rounds, unsigned long long *err,
                                    unsigned *passed, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(blocks));
    cfg.blockDim = dim3(32);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_barrier_selftest, bar, static_cast<unsigned>(blocks + missing), rounds, err,
                              passed);
}

static size_t batch_persistent_smem(int kmax, int stage) {
    return std::max(phi_counts_smem(kmax), static_cast<size_t>(kPersistWarps) * (stage + kTabScratch));
}

// 0 where the form is not offered: no room for a CTA, or K above a limit kept
// from when this launch ran the z-step too (seven documents' counts in a CTA), so
// that what was refused stays refused.
int batch_persistent_blocks_per_sm(int kmax, bool narrow, int *table_stage) {
    allow_dynamic_smem(k_batch_sweep_persistent);
    if (z_step_smem(kmax, kPersistWarps - 1, narrow) > static_cast<size_t>(smem_optin())) return 0;
    const size_t rows = static_cast<size_t>(kPersistWarps) * (dense_row_bytes(kmax) + kTabScratch);
    *table_stage = rows <= 56 * 1024 ? dense_row_bytes(kmax) : 0;       // four CTAs per SM
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_batch_sweep_persistent, kPersistThreads,
                                                      batch_persistent_smem(kmax, *table_stage)) != cudaSuccess) n = 0;
    return n;
}

cudaError_t launch_batch_sweep_persistent(const BatchLaunch &b, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(b.persist_grid));
    cfg.blockDim = dim3(kPersistThreads);
    cfg.dynamicSmemBytes = batch_persistent_smem(b.kmax, b.table_stage);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_batch_sweep_persistent, b);
    if (e != cudaSuccess) return e;
    launch_batch_z(b, st);
    return cudaGetLastError();
}

int batch_phi_blocks_per_sm(int kmax) {
    allow_dynamic_smem(k_phi_counts_multi);
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_phi_counts_multi, kPhiCountBlock, sizeof(uint32_t) * phi_count_words(kmax));
    return n > 0 ? n : 1;
}

int batch_z_blocks_per_sm(int kmax, int warps, bool narrow) {
    ZMultiKernel kern = z_multi_kernel(kmax);
    allow_dynamic_smem(kern);
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, 32 * warps, z_step_smem(kmax, warps, narrow));
    return n > 0 ? n : 1;
}

using ServeKernel = void (*)(ZArgs, ServeSlot *, const int32_t *, int, const int32_t *, int16_t *, int64_t, int *,
                            uint64_t);
static ServeKernel serve_kernel(int K) {
    switch (z_nw(K)) {
        case 1: return k_serve_step<1>;
        case 2: return k_serve_step<2>;
        case 4: return k_serve_step<4>;
        case 8: return k_serve_step<8>;
        default: return k_serve_step<0>;
    }
}

void launch_serve_step(const ZArgs &a, ServeSlot *slots, const int32_t *active, int n_active, const int32_t *arena_w,
                       int16_t *arena_z, int64_t slice, int *work, int warps_per_block, int grid, uint64_t window_ns,
                       bool narrow, cudaStream_t st) {
    if (n_active <= 0) return;
    cudaMemsetAsync(work, 0, sizeof(int), st);
    const int need = (n_active + warps_per_block - 1) / warps_per_block;
    ZArgs an = a;
    an.narrow = narrow ? 1 : 0;
    serve_kernel(a.K)<<<std::min(grid, need), 32 * warps_per_block, z_step_smem(a.K, warps_per_block, narrow), st>>>(
        an, slots, active, n_active, arena_w, arena_z, slice, work, window_ns);
}

int serve_blocks_per_sm(int K, int warps_per_block) {
    // three count planes: their shared memory bounds the launches with two
    ServeKernel kern = serve_kernel(K);
    allow_dynamic_smem(kern);
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, 32 * warps_per_block, z_step_smem(K, warps_per_block));
    return n > 0 ? n : 1;
}

void launch_doc_topic(const int64_t *doc_off, int64_t D, const int16_t *z, int K, int32_t *m_dk, cudaStream_t st) {
    if (D <= 0) return;
    cudaMemsetAsync(m_dk, 0, sizeof(int32_t) * static_cast<size_t>(D) * K, st);
    const int grid = static_cast<int>(std::min<int64_t>((D * 32 + 255) / 256, 8LL * sm_count() * 8));
    k_doc_topic<<<grid, 256, 0, st>>>(doc_off, D, z, K, m_dk);
}

void launch_n_dense(const PhiArgs &a, int32_t *n_kv, cudaStream_t st) {
    cudaMemsetAsync(n_kv, 0, sizeof(int32_t) * static_cast<size_t>(a.K) * a.V, st);
    k_n_dense<<<(a.V + 255) / 256, 256, 0, st>>>(a, n_kv);
}

void launch_phi_values(const PhiArgs &a, float *phi, cudaStream_t st) {
    k_phi_values<<<4 * sm_count(), 256, 0, st>>>(a, phi);
}

}  // namespace pulda
