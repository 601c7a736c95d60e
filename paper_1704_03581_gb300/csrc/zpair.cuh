// The z-step of two documents by one warp, sixteen lanes each, on dense rows
// (zdense.cuh) of up to 1024 topics.
//
// With a document per warp, most of a token's instructions do not depend on how
// many topics a lane owns: reading its record, its counts in and out, the scan,
// the 64-bit draw, the search.  Here each of them serves two tokens.  A lane
// owns the topics of two of the row's 32 lanes, s and s + 16 (its loads stay
// consecutive), and so has two sums: the prefix in topic order runs over the
// sixteen lanes' first sums, then over their second ones.  The sums, draws and
// topics are those of the one-document form.
// 236 warp instructions per token against 321 of the sparse walk; 99 M tokens
// at K = 1000: 32.2 ms with a document per warp, 27.8 with two (0.67 of the
// issue peak; without the accesses to the second count plane the same).
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

#include "zdense.cuh"

namespace pulda {

// Shared memory of a warp, in 32-bit words: two documents' count planes (two
// each), sixteen tokens' records each, the counters, two runs.
__host__ __device__ __forceinline__ int z_pair_words(int K) {
    return 2 * 2 * 32 * dense_words(K) + 32 * kTokRecWords + 16 + 2 * 20;
}
static_assert(sizeof(DocRun) <= 20 * sizeof(uint32_t) && (32 * kTokRecWords + 16 + 40) % 4 == 0, "a pair's areas");

// Inclusive scan of v over each half warp.
__device__ __forceinline__ u64 half_incl_scan(u64 v) { return warp_incl_scan<16>(v); }

// lane `s` of this lane's half
__device__ __forceinline__ u64 half_shfl(u64 v, int s) { return __shfl_sync(0xFFFFFFFFu, v, s, 16); }

template <int NW>
__device__ __forceinline__ u64 pair_dot(const uint8_t *row, const uint8_t *m, int l, bool wide) {
    uint32_t q[3][NW], w[NW];
#pragma unroll
    for (int p = 0; p < 3; ++p) load_words<NW>(row + p * (128 * NW), l, q[p]);
    load_words<NW>(m, l, w);
    uint32_t s0 = 0, s1 = 0, s2 = 0;
#pragma unroll
    for (int x = 0; x < NW; ++x) {
        s0 = __dp4a(w[x], q[0][x], s0);
        s1 = __dp4a(w[x], q[1][x], s1);
        s2 = __dp4a(w[x], q[2][x], s2);
    }
    u64 sum = static_cast<u64>(s0 + (s1 << 8)) + (static_cast<u64>(s2) << 16);
    if (wide) {
        load_words<NW>(m + 128 * NW, l, w);
        s0 = s1 = s2 = 0;
#pragma unroll
        for (int x = 0; x < NW; ++x) {
            s0 = __dp4a(w[x], q[0][x], s0);
            s1 = __dp4a(w[x], q[1][x], s1);
            s2 = __dp4a(w[x], q[2][x], s2);
        }
        sum += (static_cast<u64>(s0 + (s1 << 8)) + (static_cast<u64>(s2) << 16)) << 8;
    }
    return sum;
}

// Two documents (either may be empty), one pass.  r: this half's run.
template <int NW>
__device__ __forceinline__ void z_pair(const ZArgs &a, uint32_t *sm, const DocRun &r, u64 *wcnt) {
    using G = DenseGeo<NW>;
    constexpr int PB = G::PB;
    const int lane = threadIdx.x & 31, h = lane >> 4, s = lane & 15;
    const int K = a.K;
    uint8_t *m = reinterpret_cast<uint8_t *>(sm) + h * 2 * PB;
    uint4 *rec = reinterpret_cast<uint4 *>(sm + 2 * 2 * 32 * NW) + 32 * h;
    uint32_t *drow_of = sm + 2 * 2 * 32 * NW + 256 + 16 * h;
    DocRun &rs = *(reinterpret_cast<DocRun *>(wcnt + 8) + h);
    auto count = [&](int p) { return m[p] | (static_cast<uint32_t>(m[p + PB]) << 8); };
    auto set = [&](int p, uint32_t c) {
        m[p] = static_cast<uint8_t>(c);
        m[p + PB] = static_cast<uint8_t>(c >> 8);
    };
    // counts from the current topics; equal topics of a half are counted by one lane
    for (int i = s; i < 2 * PB / 16; i += 16) reinterpret_cast<uint4 *>(m)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    const int most = max(r.len, __shfl_xor_sync(0xFFFFFFFFu, r.len, 16));
    bool wide = false;
    for (int i0 = 0; i0 < most; i0 += 16) {
        const int i = i0 + s;
        const int k = i < r.len ? guard_index(r.z[i], K, a.stats) : K + h;
        const unsigned peers = __match_any_sync(0xFFFFFFFFu, k | (h << 20));
        if (i < r.len && lane == __ffs(peers) - 1) {
            const int p = G::pos(k);
            const uint32_t c = count(p) + static_cast<uint32_t>(__popc(peers));
            set(p, c);
            wide |= c > 255u;
        }
        __syncwarp();
    }
    wide = __any_sync(0xFFFFFFFFu, wide);           // either document needs the second plane
    uint32_t mb0 = 0, mb1 = 0;                      // topics with m > 0 of the row's lanes s and s + 16
#pragma unroll 1
    for (int b = 0; b < G::TPL; ++b) {
        const int p = G::lane0(b) + G::STRIDE * s;
        if (count(p)) mb0 |= 1u << b;
        if (count(p + 16 * G::STRIDE)) mb1 |= 1u << b;
    }
    int kd = __popc(mb0) + __popc(mb1);
#pragma unroll
    for (int o = 8; o; o >>= 1) kd += __shfl_xor_sync(0xFFFFFFFFu, kd, o);
    if (s == 0) rs = r;
    __syncwarp();
    const int colmax = column_limit<NW>(a.path, K);
    const int fine = s & (G::TPL - 1);
    for (int i0 = 0; i0 < most; i0 += 16) {
        const int cnt = min(16, rs.len - i0);       // this document's tokens in the block (0 or less: none)
        const int maxcnt = min(16, most - i0);
        if (s < cnt) stage_token(a, rs, i0 + s, rec + 2 * s, drow_of + s, colmax, [](int k) { return G::pos(k); });
        __syncwarp();
        int znew = 0;
        uint32_t bm0 = 0, bm1 = 0;
        if (cnt > 0) {
            bm0 = lane_bits<G::TPL>(a.bits, static_cast<int64_t>(rec[1].z) * a.KWp, s);
            bm1 = lane_bits<G::TPL>(a.bits, static_cast<int64_t>(rec[1].z) * a.KWp, s + 16);
        }
        uint32_t c_min = 0, c_cnt = 0;              // as z_doc_regs, of this half
        for (int tt = 0; tt < maxcnt; ++tt) {
            const bool act = tt < cnt;
            const uint4 t0 = rec[2 * tt], t1 = rec[2 * tt + 1];
            const int kold = act ? static_cast<int>(t1.w >> 16) : 0;
            const int n_w = static_cast<int>(t1.w & 0xFFFFu);
            const u64 At = (static_cast<u64>(t0.w) << 32) | t0.z, U = (static_cast<u64>(t1.x) << 32) | t1.y;
            const uint32_t d = act ? drow_of[tt] : 0u;
            // the token out: m^{-i} (every lane of the half stores the same bytes)
            {
                const uint32_t c = count(kold) - 1u;
                __syncwarp();
                if (act) {
                    set(kold, c);
                    if (c == 0) {
                        --kd;
                        const uint32_t bit = 1u << G::bit(kold);
                        const int o = G::owner(kold);
                        if (o == s) mb0 &= ~bit;
                        if (o == s + 16) mb1 &= ~bit;
                    }
                    c_min += static_cast<uint32_t>(kd < n_w ? kd : n_w);
                    c_cnt += (kd < n_w ? 1u : 0u) + (static_cast<uint32_t>(__popc(bm0 & mb0) + __popc(bm1 & mb1)) << 18);
                }
                __syncwarp();
            }
            if (tt + 1 < cnt) {
                const int64_t wrow = static_cast<int64_t>(rec[2 * tt + 3].z) * a.KWp;
                bm0 = lane_bits<G::TPL>(a.bits, wrow, s);
                bm1 = lane_bits<G::TPL>(a.bits, wrow, s + 16);
            }
            // This half's sums: over its word's column when that is short or
            // there is no row (the lane's share of its entries, as the first
            // sum), else over the row's lanes s and s + 16.
            const bool cols = d == 0xFFFFFFFFu;
            const int64_t col = static_cast<int64_t>((static_cast<u64>(t0.y & 0xFFFFu) << 32) | t0.x);
            const int seg = (n_w + 15) >> 4;
            const uint8_t *row = a.qrow + static_cast<size_t>(cols ? 0u : d) * (3 * PB);
            u64 sa = 0, sb = 0;
            if (cols) {
                const int j1 = min(seg * s + seg, n_w);
#pragma unroll 2
                for (int j = seg * s; j < j1; ++j)
                    sa += static_cast<u64>(a.q[col + j]) * count(G::pos(guard_index(a.topic[col + j], K, a.stats)));
            } else {
                sa = pair_dot<NW>(row, m, s, wide);
                sb = pair_dot<NW>(row, m, s + 16, wide);
            }
            __syncwarp();
            const u64 ia = half_incl_scan(sa), ib = half_incl_scan(sb);
            const u64 ta = half_shfl(ia, 15);
            const u64 T = At + ((ta + half_shfl(ib, 15)) << kFracBits);
            u64 rb = (__umul64hi(U, T) - At) >> kFracBits;
            const int half = rb < ta ? 0 : 16;      // an alias draw's rb passes both
            rb -= half ? ta : 0ull;
            const u64 sum = half ? sb : sa, incl = half ? ib : ia;
            const uint32_t bal = (__ballot_sync(0xFFFFFFFFu, rb < incl) >> (16 * h)) & 0xFFFFu;
            const bool settled = bal == 0;          // the alias table's outcome, or no mass at all
            const int L = (__ffs(bal) - 1) & 15;
            const u64 res = half_shfl(rb - (incl - sum), L);
            const uint32_t hi = __shfl_sync(0xFFFFFFFFu, static_cast<uint32_t>(sum >> 32), L, 16);
            // the found lane's terms, one or two a lane of this half: its
            // column entries, or its topics
            uint32_t knew = 0xFFFFFFFFu;
            uint32_t q0 = 0, q1 = 0;
            int p0 = 0, p1 = 0;
            if (cols) {
                const int j = seg * L + s;
                if (s < seg && j < n_w) {
                    q0 = a.q[col + j];
                    p0 = G::pos(guard_index(a.topic[col + j], K, a.stats));
                }
            } else {
                auto weight = [&](int p) {
                    return row[p] | (static_cast<uint32_t>(row[p + PB]) << 8) | (static_cast<uint32_t>(row[p + 2 * PB]) << 16);
                };
                p0 = G::lane0(fine) + (L + half) * G::STRIDE;
                if (NW == 8 || s < G::TPL) q0 = weight(p0);
                if (NW == 8) {
                    p1 = p0 + 512;
                    q1 = weight(p1);
                }
            }
            __syncwarp();
            const uint32_t n0 = count(p0), n1 = NW == 8 ? count(p1) : 0u;
            uint32_t f0, f1 = 0;
            if (!__any_sync(0xFFFFFFFFu, hi != 0)) {
                const uint32_t r32 = static_cast<uint32_t>(res);
                const uint32_t x0 = warp_incl_scan<16>(q0 * n0);
                f0 = __ballot_sync(0xFFFFFFFFu, r32 < x0);
                if (NW == 8) f1 = __ballot_sync(0xFFFFFFFFu, r32 < warp_incl_scan<16>(q1 * n1) + __shfl_sync(0xFFFFFFFFu, x0, 15, 16));
            } else {
                const u64 x0 = half_incl_scan(static_cast<u64>(q0) * n0);
                f0 = __ballot_sync(0xFFFFFFFFu, res < x0);
                if (NW == 8) f1 = __ballot_sync(0xFFFFFFFFu, res < half_incl_scan(static_cast<u64>(q1) * n1) + half_shfl(x0, 15));
            }
            f0 = (f0 >> (16 * h)) & 0xFFFFu;
            f1 = (f1 >> (16 * h)) & 0xFFFFu;
            const int at0 = __shfl_sync(0xFFFFFFFFu, p0, (__ffs(f0) - 1) & 15, 16);
            const int at1 = NW == 8 ? __shfl_sync(0xFFFFFFFFu, p1, (__ffs(f1) - 1) & 15, 16) : 0;
            if (f0 | f1) knew = static_cast<uint32_t>(f0 ? at0 : at1);
            if (__any_sync(0xFFFFFFFFu, cols && seg > 16)) {
                // a long column (a word without a row): its found lane walks the share
                int f = -1;
                if (cols && seg > 16 && s == L && !settled) {
                    u64 run = 0;
                    const int j1 = min(seg * s + seg, n_w);
                    for (int j = seg * s; j < j1; ++j) {
                        const int k = G::pos(guard_index(a.topic[col + j], K, a.stats));
                        run += static_cast<u64>(a.q[col + j]) * count(k);
                        if (res < run) { f = k; break; }
                    }
                }
                f = __shfl_sync(0xFFFFFFFFu, f, L, 16);
                if (cols && seg > 16) knew = static_cast<uint32_t>(f);
            }
            if (settled) {
                const bool none = T == 0;
                knew = none ? static_cast<uint32_t>(kold) : t0.y >> 16;
                if (act) c_cnt += none ? 1u << 12 : 1u << 6;
            } else if (act && knew == 0xFFFFFFFFu) {
                if (s == 0) atomicOr(&a.stats[ST_ERROR], ERR_INTERNAL);
                knew = static_cast<uint32_t>(kold);
            }
            if (!act) knew = 0;
            // back in with its new topic
            {
                const uint32_t c = count(static_cast<int>(knew)) + 1u;
                __syncwarp();
                if (act) {
                    set(static_cast<int>(knew), c);
                    if (c == 1) {
                        ++kd;
                        const uint32_t bit = 1u << G::bit(static_cast<int>(knew));
                        const int o = G::owner(static_cast<int>(knew));
                        if (o == s) mb0 |= bit;
                        if (o == s + 16) mb1 |= bit;
                    }
                }
                if (!wide) wide = __any_sync(0xFFFFFFFFu, act && c == 256u);
            }
            if (s == tt) znew = static_cast<int>(knew);
        }
        if (s < cnt) rs.z[i0 + s] = static_cast<int16_t>(guard_index(G::topic(znew), K, a.stats));
        {
            // the block's counts of both documents into the warp's counters
            const uint32_t mine = static_cast<uint32_t>(max(cnt, 0));
            const uint32_t jsum = __reduce_add_sync(0xFFFFFFFFu, c_cnt >> 18);
            auto both = [](uint32_t v) { return v + __shfl_xor_sync(0xFFFFFFFFu, v, 16); };
            const uint32_t tok = both(mine), mn = both(c_min), packed = both(c_cnt & 0x3FFFFu);
            const uint32_t v = lane == 0 ? tok : lane == 1 ? (packed >> 6) & 63u : lane == 2 ? mn
                             : lane == 3 ? (packed >> 12) & 63u : lane == 4 ? jsum : packed & 63u;
            if (lane < 6) wcnt[lane] += v;
        }
        __syncwarp();
    }
}

}  // namespace pulda
