// The z-step of one document by one warp, on dense byte-plane rows.
//
// Per token the sampler needs B = sum_k q_{k,v} m_k over the document's
// topics and, when the draw lands in that part, the topic where the running
// sum passes it.  Walking the intersection of two sparse sets costs a chain
// of dependent loads and uneven work per lane.  Here the word's fixed-point
// weights q (24 bits) lie as three planes of bytes and the document's counts
// m as planes of bytes, in the same topic order, so that one dp4a multiplies
// and adds four topics: 24 dp4a per lane cover 1024 topics, the row's loads
// do not depend on the document's state (the next token's row is fetched
// while this one is drawn), and no lane waits on a busier one.  All sums are
// the exact integers of the sparse walk, so every draw is the same.
// What bounds it: instruction issue and the L1 data pipe where many documents
// run (K = 1000, 99 M tokens: 34.5 ms for the sparse walk, 32.2 for this;
// 12.4 M tokens 8.3 and 4.0 with the longest documents on CTAs), latency
// where few do.
//
// Layout (pulda_internal.h): lane l owns the TPL = 4 NW consecutive topics
// [TPL l, TPL l + TPL); topic k's byte lies at dense_pos(k) of each plane.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

#include "checks.cuh"
#include "device_rng.cuh"
#include "pulda_internal.h"
#include "zstep.cuh"

namespace pulda {

// Inclusive scans over aligned segments of W lanes.  The shuffle's own
// predicate (source lane in the segment) guards the add, so a step is two
// instructions (64 bits: four).
template <int W = 32>
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x) {
#pragma unroll
    for (int o = 1; o < W; o <<= 1)
        asm volatile("{ .reg .u32 t; .reg .pred p; shfl.sync.up.b32 t|p, %0, %1, %2, 0xffffffff; @p add.u32 %0, %0, t; }"
                     : "+r"(x) : "r"(o), "n"((32 - W) << 8));
    return x;
}
template <int W = 32>
__device__ __forceinline__ u64 warp_incl_scan(u64 v) {
    uint32_t lo = static_cast<uint32_t>(v), hi = static_cast<uint32_t>(v >> 32);
#pragma unroll
    for (int o = 1; o < W; o <<= 1)
        asm volatile("{ .reg .u32 a, b; .reg .pred p; shfl.sync.up.b32 a|p, %0, %2, %3, 0xffffffff;\n\t"
                     "shfl.sync.up.b32 b, %1, %2, %3, 0xffffffff;\n\t"
                     "@p add.cc.u32 %0, %0, a;\n\t@p addc.u32 %1, %1, b; }"
                     : "+r"(lo), "+r"(hi) : "r"(o), "n"((32 - W) << 8));
    return (static_cast<u64>(hi) << 32) | lo;
}

// The counts of one document in a warp's shared memory: plane p's byte at
// dense_pos(k) is bits [8p, 8p + 8) of topic k's count.  `lvl` (the same in
// every lane) is the highest plane that may hold a nonzero byte: planes above
// it are neither read nor written, so a document whose topics stay below 256
// tokens touches one plane.
struct DocCounts {
    uint8_t *b;
    int PB;         // bytes of a plane
    int lvl;
    __device__ __forceinline__ uint32_t get(int pos) const {
        uint32_t c = b[pos];
        if (lvl > 0) {
            c |= static_cast<uint32_t>(b[PB + pos]) << 8;
            if (lvl > 1) c |= static_cast<uint32_t>(b[2 * PB + pos]) << 16;
        }
        return c;
    }
    // writes the planes up to the larger of lvl and c's own
    __device__ __forceinline__ void set(int pos, uint32_t c) {
        b[pos] = static_cast<uint8_t>(c);
        if (lvl > 0 || c > 0xFFu) {
            b[PB + pos] = static_cast<uint8_t>(c >> 8);
            if (lvl > 1 || c > 0xFFFFu) b[2 * PB + pos] = static_cast<uint8_t>(c >> 16);
        }
    }
};

__device__ __forceinline__ int count_level(uint32_t c) { return (c > 0xFFu ? 1 : 0) + (c > 0xFFFFu ? 1 : 0); }

// Fills the counts of a run's topics (or, with m0, from those K counts) and
// sets lvl.  Tokens 32 at a time: equal topics are counted by one lane, so no
// byte is added to by two lanes and none carries into its neighbour.
template <typename Pos>
__device__ __forceinline__ void build_counts(const ZArgs &a, DocCounts &m, const DocRun &r, const uint32_t *m0, int planes, Pos pos) {
    const int lane = threadIdx.x & 31;
    uint4 *z = reinterpret_cast<uint4 *>(m.b);
    for (int i = lane; i < planes * m.PB / 16; i += 32) z[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    m.lvl = planes - 1;
    int top = 0;
    if (m0) {
        for (int k = lane; k < a.K; k += 32) {
            const uint32_t c = m0[k];
            if (c) m.set(pos(k), c);
            top = max(top, count_level(c));
        }
    } else {
        for (int i0 = 0; i0 < r.len; i0 += 32) {
            const int i = i0 + lane;
            const int k = i < r.len ? guard_index(r.z[i], a.K, a.stats) : -1;
            const unsigned peers = __match_any_sync(0xFFFFFFFFu, k);
            if (k >= 0 && lane == __ffs(peers) - 1) {
                const int p = pos(k);
                const uint32_t c = m.get(p) + static_cast<uint32_t>(__popc(peers));
                m.set(p, c);
                top = max(top, count_level(c));
            }
            __syncwarp();
        }
    }
    m.lvl = static_cast<int>(__reduce_max_sync(0xFFFFFFFFu, static_cast<unsigned>(top)));
    __syncwarp();
}

// Which of the sixteen topics from position p on (one chunk of a lane) have m > 0.
__device__ __forceinline__ uint32_t nonzero_topics(const DocCounts &m, int p, int planes) {
    uint4 v = *reinterpret_cast<const uint4 *>(m.b + p);
    for (int pl = 1; pl < planes; ++pl) {
        const uint4 u = *reinterpret_cast<const uint4 *>(m.b + p + pl * m.PB);
        v = make_uint4(v.x | u.x, v.y | u.y, v.z | u.z, v.w | u.w);
    }
    auto four = [](uint32_t x) { return ((__vcmpne4(x, 0u) & 0x01010101u) * 0x01020408u) >> 24 & 15u; };
    return four(v.x) | four(v.y) << 4 | four(v.z) << 8 | four(v.w) << 12;
}

// NW words of a plane (bytes of this lane's topics) from p, one to eight.
template <int NW>
__device__ __forceinline__ void load_words(const uint8_t *p, int lane, uint32_t (&w)[NW]) {
    if constexpr (NW == 1) {
        w[0] = *reinterpret_cast<const uint32_t *>(p + 4 * lane);
    } else if constexpr (NW == 2) {
        const uint2 v = *reinterpret_cast<const uint2 *>(p + 8 * lane);
        w[0] = v.x; w[1] = v.y;
    } else {
#pragma unroll
        for (int c = 0; c < NW / 4; ++c) {
            const uint4 v = *reinterpret_cast<const uint4 *>(p + 512 * c + 16 * lane);
            w[4 * c] = v.x; w[4 * c + 1] = v.y; w[4 * c + 2] = v.z; w[4 * c + 3] = v.w;
        }
    }
}

// Geometry of the register form (K <= 1024): NW words per lane and plane.
// The token loop names a topic by its position in a plane.
template <int NW>
struct DenseGeo {
    static constexpr int TPL = 4 * NW;
    static constexpr int PB = 128 * NW;
    __device__ static __forceinline__ int pos(int k) { return NW == 8 ? ((k & 16) << 5) | ((k >> 5) << 4) | (k & 15) : k; }
    __device__ static __forceinline__ int topic(int pos) { return NW == 8 ? ((pos & 512) >> 5) | ((pos & 496) << 1) | (pos & 15) : pos; }
    // lane and bit (of its TPL) that own a position
    __device__ static __forceinline__ int owner(int pos) { return NW == 8 ? (pos >> 4) & 31 : pos / TPL; }
    __device__ static __forceinline__ int bit(int pos) { return NW == 8 ? ((pos >> 9) << 4) | (pos & 15) : pos % TPL; }
    // position of lane 0's topic t; lane l's is 16 (NW = 8) or TPL bytes per lane further on
    __device__ static __forceinline__ int lane0(int t) { return NW == 8 ? ((t & 16) << 5) | (t & 15) : t; }
    static constexpr int STRIDE = NW == 8 ? 16 : TPL;
};

// The lane's sum of q m over its topics.
template <int NW>
__device__ __forceinline__ u64 dense_dot(const uint32_t (&q)[3][NW], const DocCounts &m, int lane) {
    u64 sum = 0;
    for (int p = 0; p <= m.lvl; ++p) {
        uint32_t w[NW];
        load_words<NW>(m.b + p * (128 * NW), lane, w);
        uint32_t s0 = 0, s1 = 0, s2 = 0;        // at most 32 topics of 255^2 each
#pragma unroll
        for (int x = 0; x < NW; ++x) {
            s0 = __dp4a(w[x], q[0][x], s0);
            s1 = __dp4a(w[x], q[1][x], s1);
            s2 = __dp4a(w[x], q[2][x], s2);
        }
        sum += (static_cast<u64>(s0 + (s1 << 8)) + (static_cast<u64>(s2) << 16)) << (8 * p);
    }
    return sum;
}

// Lane j's prefix of q m over the first j + 1 topics of a group (its bytes
// at off of every plane; lanes past the group repeat it): the counts of the
// later topics are masked off.  Every lane reads the same words.
template <int GW>
__device__ __forceinline__ u64 group_prefix(const uint8_t *row, int PB, const DocCounts &m, int off, int lane) {
    const int j = lane & (4 * GW - 1);
    uint32_t mask[GW];
#pragma unroll
    for (int x = 0; x < GW; ++x) {
        const int t = j - 4 * x;                        // last topic of word x that counts
        mask[x] = t >= 3 ? 0xFFFFFFFFu : t < 0 ? 0u : (1u << (8 * (t & 3) + 8)) - 1u;
    }
    uint32_t q[3][GW];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        if constexpr (GW == 2) {
            const uint2 v = *reinterpret_cast<const uint2 *>(row + p * PB + off);
            q[p][0] = v.x; q[p][1] = v.y;
        } else {
            q[p][0] = *reinterpret_cast<const uint32_t *>(row + p * PB + off);
        }
    }
    u64 sum = 0;
    for (int pl = 0; pl <= m.lvl; ++pl) {
        uint32_t s0 = 0, s1 = 0, s2 = 0;
#pragma unroll
        for (int x = 0; x < GW; ++x) {
            const uint32_t w = *reinterpret_cast<const uint32_t *>(m.b + pl * PB + off + 4 * x) & mask[x];
            s0 = __dp4a(w, q[0][x], s0);
            s1 = __dp4a(w, q[1][x], s1);
            s2 = __dp4a(w, q[2][x], s2);
        }
        sum += (static_cast<u64>(s0 + (s1 << 8)) + (static_cast<u64>(s2) << 16)) << (8 * pl);
    }
    return sum;
}

// What one token's draw needs besides the sums.
struct TokenDraw {
    u64 At, U;
    int ka, kold;       // the alias outcome and the current topic
};

// The draw r = floor(u (A + 2^16 B)): the alias outcome when r < A, else the
// remaining mass rb in units of q.  Returns the topic when it is settled, -1
// when rb picks it.
__device__ __forceinline__ int split_draw(const TokenDraw &t, u64 B, u64 &rb, uint32_t &c_cnt) {
    const u64 T = t.At + (B << kFracBits);
    if (T == 0) {
        c_cnt += 1u << 12;
        return t.kold;
    }
    const u64 rr = __umul64hi(t.U, T);
    if (rr < t.At) {
        c_cnt += 1u << 6;
        return t.ka;
    }
    rb = (rr - t.At) >> kFracBits;
    return -1;
}

// First lane of a segment of W lanes, holding consecutive topics, whose
// running sum of q m passes res; W when none does.
template <int W, typename S>
__device__ __forceinline__ int fine_search(S p, S res) {
    const uint32_t f = __ballot_sync(0xFFFFFFFFu, res < warp_incl_scan<W>(p));
    return f ? __ffs(f) - 1 : W;
}

// The new topic (position) from the lanes' sums of q m: the lane whose prefix
// passes the draw, then its TPL topics, one per lane.
template <int NW>
__device__ __forceinline__ int dense_draw(const ZArgs &a, u64 sum, const TokenDraw &t, const uint8_t *row, const DocCounts &m,
                                          int fine, uint32_t &c_cnt) {
    using G = DenseGeo<NW>;
    constexpr int W = G::TPL;
    const u64 incl = warp_incl_scan<32>(sum);
    u64 rb;
    const int settled = split_draw(t, __shfl_sync(0xFFFFFFFFu, incl, 31), rb, c_cnt);
    if (settled >= 0) return settled;
    const int L = __ffs(__ballot_sync(0xFFFFFFFFu, rb < incl)) - 1;      // rb < B: some lane passes it
    const u64 res = __shfl_sync(0xFFFFFFFFu, rb - (incl - sum), L);
    const int at = fine + L * G::STRIDE;                                 // this lane's topic of lane L's
    const uint32_t q = row[at] | (static_cast<uint32_t>(row[at + G::PB]) << 8) | (static_cast<uint32_t>(row[at + 2 * G::PB]) << 16);
    const u64 p = static_cast<u64>(q) * m.get(at);
    // lane L's topics sum to less than 2^32 but for counts in the hundreds
    const int f = __shfl_sync(0xFFFFFFFFu, static_cast<uint32_t>(sum >> 32), L) == 0
                      ? fine_search<W, uint32_t>(static_cast<uint32_t>(p), static_cast<uint32_t>(res))
                      : fine_search<W, u64>(p, res);
    if (f >= W) {
        if ((threadIdx.x & 31) == 0) atomicOr(&a.stats[ST_ERROR], ERR_INTERNAL);
        return t.kold;
    }
    return G::lane0(f) + L * G::STRIDE;
}

// The same over the word's column (words with few topics, or without a dense
// row): lane l takes a contiguous share of its n_w entries, B of them loaded at
// once; a found lane's share of more than B is shared out, an entry per lane (a
// lane that walked it waited on a load per entry).
template <int B, typename Pos>
__device__ __forceinline__ int column_draw(const ZArgs &a, const TokenDraw &t, int64_t col, int n_w, const DocCounts &m,
                                           int lane, uint32_t &c_cnt, Pos pos) {
    __syncwarp();                                        // the column reads every lane's counts
    const int seg = (n_w + 31) >> 5;
    const int j0 = min(seg * lane, n_w), j1 = min(j0 + seg, n_w);
    u64 acc = 0, term[B];
    int at[B];
    for (int j = j0; j == j0 || j < j1; j += B) {
        uint32_t q[B];
        int k[B];
#pragma unroll
        for (int i = 0; i < B; ++i) {
            q[i] = j + i < j1 ? a.q[col + j + i] : 0u;
            k[i] = j + i < j1 ? a.topic[col + j + i] : 0;
        }
#pragma unroll
        for (int i = 0; i < B; ++i) {
            at[i] = pos(guard_index(k[i], a.K, a.stats));
            term[i] = static_cast<u64>(q[i]) * m.get(at[i]);
            acc += term[i];
        }
    }
    const u64 incl = warp_incl_scan(acc);
    u64 rb;
    const int settled = split_draw(t, __shfl_sync(0xFFFFFFFFu, incl, 31), rb, c_cnt);
    if (settled >= 0) return settled;
    const int L = __ffs(__ballot_sync(0xFFFFFFFFu, rb < incl)) - 1;
    u64 res = __shfl_sync(0xFFFFFFFFu, rb - (incl - acc), L);
    if (seg <= B) {
        int f = -1;
        u64 upto = acc;
#pragma unroll
        for (int i = B - 1; i >= 0; --i) {
            if (res < upto) f = at[i];
            upto -= term[i];
        }
        f = __shfl_sync(0xFFFFFFFFu, f, L);
        if (f >= 0) return f;
    }
    const int end = min(seg * L + seg, n_w);
    for (int i0 = seg <= B ? end : seg * L; i0 < end; i0 += 32) {
        const int j = i0 + lane;
        const int k = pos(guard_index(j < end ? a.topic[col + j] : 0, a.K, a.stats));
        const u64 p = j < end ? static_cast<u64>(a.q[col + j]) * m.get(k) : 0;
        const u64 upto = warp_incl_scan(p);
        const uint32_t f = __ballot_sync(0xFFFFFFFFu, res < upto);
        if (f) return __shfl_sync(0xFFFFFFFFu, k, __ffs(f) - 1);
        res -= __shfl_sync(0xFFFFFFFFu, upto, 31);
    }
    if (lane == 0) atomicOr(&a.stats[ST_ERROR], ERR_INTERNAL);
    return t.kold;
}

// A word with at most this many nonzero topics is summed over its column
// even when it has a dense row: one or two entries per lane instead of the
// whole row, which for such (rare) words mostly comes from beyond L1.  Above
// 1,024 topics a row's work grows with K: with a limit of 128, K / 16, K / 10 and
// K / 6 a pass over 12,000 documents of 200 tokens, one per warp, takes 3.2, 3.1,
// 3.0 and 3.0 ms at K = 3,000, 6.5, 5.5, 5.3 and 5.5 at 8,000, 24.8, 16.5, 16.1 and
// 16.2 at 16,384.
// zstep_path 1 raises the limit, 2 takes the row wherever there is one.
template <int NW>
__device__ __forceinline__ constexpr int column_max() { return NW == 0 ? 128 : NW == 8 ? 64 : NW == 4 ? 32 : 0; }
template <int NW>
__device__ __forceinline__ int column_limit(int path, int K) {
    const int most = NW > 0 ? column_max<NW>() : max(column_max<NW>(), K / 10);
    return path == 1 ? 2 * most + 32 : path == 2 ? -1 : most;
}

// The staging records of a warp: where z_doc keeps them for its K.
template <int NW>
__device__ __forceinline__ uint4 *token_records(uint32_t *sm, const ZArgs &a) {
    return reinterpret_cast<uint4 *>(sm + z_dense_count_words(a.K, a.narrow != 0));
}

// This block's counters (see z_doc) into the warp's, lane j its counter j.
__device__ __forceinline__ void add_block_counts(u64 *wcnt, int lane, int cnt, uint32_t c_min, uint32_t c_cnt, uint32_t c_int) {
    const uint32_t jsum = __reduce_add_sync(0xFFFFFFFFu, c_int);
    const uint32_t v = lane == 0 ? static_cast<uint32_t>(cnt)
                     : lane == 1 ? (c_cnt >> 6) & 63u
                     : lane == 2 ? c_min
                     : lane == 3 ? (c_cnt >> 12) & 63u
                     : lane == 4 ? jsum : c_cnt & 63u;
    if (lane < 6) wcnt[lane] += v;
}

// The tokens of one 32-token block, in order.  Every lane carries out the
// count updates (the same byte, the same value), so they need neither a branch
// nor a vote.
template <int NW>
__device__ __forceinline__ int z_block(const ZArgs &a, DocCounts &m, const uint4 *rec, const uint32_t *drow_of, int cnt,
                                       uint32_t &mbits, int &kd, uint32_t &c_min, uint32_t &c_cnt) {
    using G = DenseGeo<NW>;
    const int lane = threadIdx.x & 31;
    const int fine = G::lane0(lane & (G::TPL - 1));
    int znew = 0;
    uint32_t q[3][NW];
    const uint8_t *row = nullptr;
    auto fetch_row = [&](uint32_t d) {
        if (d == 0xFFFFFFFFu) return;
        row = a.qrow + static_cast<size_t>(d) * (3 * G::PB);
#pragma unroll
        for (int p = 0; p < 3; ++p) load_words<NW>(row + p * G::PB, lane, q[p]);
    };
    uint32_t d = drow_of[0];
    fetch_row(d);
    uint32_t bm = lane_bits<G::TPL>(a.bits, static_cast<int64_t>(rec[1].z) * a.KWp, lane);
    for (int tt = 0; tt < cnt; ++tt) {
        const uint4 t0 = rec[2 * tt], t1 = rec[2 * tt + 1];
        TokenDraw t;
        t.kold = static_cast<int>(t1.w >> 16);
        const int n_w = static_cast<int>(t1.w & 0xFFFFu);
        t.At = (static_cast<u64>(t0.w) << 32) | t0.z;
        t.U = (static_cast<u64>(t1.x) << 32) | t1.y;
        t.ka = static_cast<int>(t0.y >> 16);
        // remove the token: m^{-i}
        {
            const uint32_t c = m.get(t.kold) - 1u;
            __syncwarp();
            m.set(t.kold, c);
            if (c == 0) {
                --kd;
                if (lane == G::owner(t.kold)) mbits &= ~(1u << G::bit(t.kold));
            }
        }
        c_min += static_cast<uint32_t>(kd < n_w ? kd : n_w);
        c_cnt += (kd < n_w ? 1u : 0u) + (static_cast<uint32_t>(__popc(bm & mbits)) << 18);
        const bool more = tt + 1 < cnt;
        if (more) bm = lane_bits<G::TPL>(a.bits, static_cast<int64_t>(rec[2 * tt + 3].z) * a.KWp, lane);
        const uint32_t dn = more ? drow_of[tt + 1] : 0xFFFFFFFFu;
        int knew;
        if (d != 0xFFFFFFFFu) {
            const u64 sum = dense_dot<NW>(q, m, lane);
            const uint8_t *r0 = row;
            fetch_row(dn);                  // the next token's row, while this one is drawn
            knew = dense_draw<NW>(a, sum, t, r0, m, fine, c_cnt);
        } else {
            const int64_t col = static_cast<int64_t>((static_cast<u64>(t0.y & 0xFFFFu) << 32) | t0.x);
            knew = column_draw<2>(a, t, col, n_w, m, lane, c_cnt, [](int k) { return G::pos(k); });
            fetch_row(dn);
        }
        d = dn;
        // add it back with its new topic
        {
            const uint32_t c = m.get(knew) + 1u;
            __syncwarp();
            m.set(knew, c);
            if (c == 256u || c == 65536u) m.lvl = max(m.lvl, count_level(c));
            if (c == 1) {
                ++kd;
                if (lane == G::owner(knew)) mbits |= 1u << G::bit(knew);
            }
        }
        if (lane == tt) znew = knew;
    }
    return znew;
}

// Resamples the tokens of one document, by one warp, in position order, pass
// after pass, until `budget` tokens are done or `max_pass_end` passes have
// been completed.  The counts are rebuilt from the current topics first: with
// positions < pos already resampled in this pass they are exactly those of the
// sequential sampler at `pos`.  With m0 set they start from those K counts (a
// slice of a longer document).  Returns the run's final (sweep, pos) through
// r.  sm: the warp's z_dense_warp_words(K, narrow) words, 16-byte aligned.
template <int NW>
__device__ __forceinline__ void z_doc_regs(const ZArgs &a, uint32_t *sm, DocRun &r, u64 *wcnt, const uint32_t *m0) {
    using G = DenseGeo<NW>;
    const int lane = threadIdx.x & 31;
    if (r.len == 0 || r.budget <= 0) return;
    DocCounts m{reinterpret_cast<uint8_t *>(sm), G::PB, 0};
    build_counts(a, m, r, m0, z_count_planes(a.narrow != 0), [](int k) { return G::pos(k); });
    uint32_t mbits = 0;         // this lane's topics with m > 0
#pragma unroll 1
    for (int b = 0; b < G::TPL; ++b)
        if (m.get(G::lane0(b) + G::STRIDE * lane) > 0) mbits |= 1u << b;
    int kd = static_cast<int>(__reduce_add_sync(0xFFFFFFFFu, static_cast<unsigned>(__popc(mbits))));
    // the run's state lives in shared memory while its tokens are drawn
    DocRun &rs = *z_warp_run(wcnt);
    if (lane == 0) rs = r;
    __syncwarp();
    uint4 *rec = token_records<NW>(sm, a);
    uint32_t *drow_of = reinterpret_cast<uint32_t *>(rec + 64);
    const uint32_t sweep_end = rs.sweep + static_cast<uint32_t>(rs.max_pass_end);
    const int colmax = column_limit<NW>(a.path, a.K);
    bool first = true;
    while (rs.budget > 0 && rs.sweep != sweep_end) {
        if (rs.deadline != ~0ull && !first) {
            uint64_t now = 0;
            if (lane == 0) now = global_ns();
            if (__shfl_sync(0xFFFFFFFFu, now, 0) >= rs.deadline) break;
        }
        first = false;
        const int i0 = rs.pos;
        const int cnt = static_cast<int>(min(static_cast<int64_t>(32), min(static_cast<int64_t>(rs.len - i0), rs.budget)));
        if (lane < cnt) stage_token(a, rs, i0 + lane, rec + 2 * lane, drow_of + lane, colmax, [](int k) { return G::pos(k); });
        __syncwarp();
        // this block's counters, in 32 bits: c_min = sum of min(K_d, K_v); in
        // c_cnt tokens with K_d < K_v in bits 0-5, alias draws in 6-11,
        // zero-mass tokens in 12-17 (each at most 32), this lane's share of
        // |J| (at most 32 x 32) from bit 18
        uint32_t c_min = 0, c_cnt = 0;
        const int znew = z_block<NW>(a, m, rec, drow_of, cnt, mbits, kd, c_min, c_cnt);
        if (lane < cnt) rs.z[i0 + lane] = static_cast<int16_t>(guard_index(G::topic(znew), a.K, a.stats));
        add_block_counts(wcnt, lane, cnt, c_min, c_cnt, c_cnt >> 18);
        __syncwarp();
        if (lane == 0) {
            rs.budget -= cnt;
            rs.pos += cnt;
            if (rs.pos == rs.len) { rs.pos = 0; rs.sweep += 1; }
        }
        __syncwarp();
    }
    r = rs;
    __syncwarp();
}

// K > 1024: this lane's sum over its C chunks of one count plane (at most 512
// topics of 255^2 each).
__device__ __forceinline__ u64 big_plane_dot(const uint8_t *row, const uint8_t *plane, int PB, int C, int lane) {
    uint32_t s0 = 0, s1 = 0, s2 = 0;
    const uint8_t *mp = plane + 16 * lane, *rp = row + 16 * lane;
#pragma unroll 2
    for (int c = 0; c < C; ++c) {
        const uint4 w = *reinterpret_cast<const uint4 *>(mp + 512 * c);
        const uint4 a0 = *reinterpret_cast<const uint4 *>(rp + 512 * c);
        const uint4 a1 = *reinterpret_cast<const uint4 *>(rp + 512 * c + PB);
        const uint4 a2 = *reinterpret_cast<const uint4 *>(rp + 512 * c + 2 * PB);
        s0 = __dp4a(w.x, a0.x, s0); s1 = __dp4a(w.x, a1.x, s1); s2 = __dp4a(w.x, a2.x, s2);
        s0 = __dp4a(w.y, a0.y, s0); s1 = __dp4a(w.y, a1.y, s1); s2 = __dp4a(w.y, a2.y, s2);
        s0 = __dp4a(w.z, a0.z, s0); s1 = __dp4a(w.z, a1.z, s1); s2 = __dp4a(w.z, a2.z, s2);
        s0 = __dp4a(w.w, a0.w, s0); s1 = __dp4a(w.w, a1.w, s1); s2 = __dp4a(w.w, a2.w, s2);
    }
    return static_cast<u64>(s0) + (static_cast<u64>(s1) << 8) + (static_cast<u64>(s2) << 16);
}

// U chunks of a row from chunk c0 on, and their sum over planes 0 to lvl: for
// few documents at a time, where nothing else hides a load.
template <int U>
__device__ __forceinline__ void big_load(const uint8_t *row, int PB, int C, int c0, int lane, uint4 (&q)[U][3]) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int p = 0; p < 3; ++p)
            q[u][p] = c0 + u < C ? *reinterpret_cast<const uint4 *>(row + 16 * lane + 512 * (c0 + u) + p * PB) : make_uint4(0u, 0u, 0u, 0u);
}
template <int U>
__device__ __forceinline__ u64 big_dot(const uint4 (&q)[U][3], const DocCounts &m, int PB, int C, int c0, int lane) {
    u64 acc = 0;
#pragma unroll 1
    for (int pl = 0; pl <= m.lvl; ++pl) {
        uint32_t s[3] = {0, 0, 0};
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (c0 + u >= C) continue;
            const uint4 w = *reinterpret_cast<const uint4 *>(m.b + 16 * lane + pl * PB + 512 * (c0 + u));
#pragma unroll
            for (int p = 0; p < 3; ++p)
                s[p] = __dp4a(w.w, q[u][p].w, __dp4a(w.z, q[u][p].z, __dp4a(w.y, q[u][p].y, __dp4a(w.x, q[u][p].x, s[p]))));
        }
        acc += (static_cast<u64>(s[0]) + (static_cast<u64>(s[1]) << 8) + (static_cast<u64>(s[2]) << 16)) << (8 * pl);
    }
    return acc;
}

// K > 1024: the topic of lane L's 16 C whose running sum passes res (position,
// or -1): its 2 C groups of eight, one per lane, then the group's topics.
__device__ __forceinline__ int big_find(int L, u64 res, const uint8_t *row, const DocCounts &m, int PB, int C, int lane) {
    int grp = -1;
    for (int g0 = 0; g0 < 2 * C; g0 += 32) {
        const int gi = g0 + lane;
        u64 gs = 0;
        if (gi < 2 * C) gs = group_prefix<2>(row, PB, m, ((gi >> 1) << 9) + (L << 4) + ((gi & 1) << 3), 7);
        const u64 gin = warp_incl_scan<32>(gs);
        const uint32_t f = __ballot_sync(0xFFFFFFFFu, res < gin);
        if (f) {
            const int l2 = __ffs(f) - 1;
            res = __shfl_sync(0xFFFFFFFFu, res - (gin - gs), l2);
            grp = g0 + l2;
            break;
        }
        res -= __shfl_sync(0xFFFFFFFFu, gin, 31);
    }
    if (grp < 0) return -1;
    const int off = ((grp >> 1) << 9) + (L << 4) + ((grp & 1) << 3);
    const u64 p = group_prefix<2>(row, PB, m, off, lane);
    const uint32_t f = __ballot_sync(0xFFFFFFFFu, res < p) & 0xFFu;
    return f ? off + __ffs(f) - 1 : -1;
}

// The same for K > 1024: 512 C topics, lane l owning the 16 C from 16 C l on,
// in C chunks of one 16-byte load per plane.  A lane holds no row and no
// group sums: it accumulates its chunks, and the found lane's 2 C groups of
// eight topics are summed again, one group per lane.  The topics that document and
// word share are counted over words in topic order, 16 bytes a lane (over every
// lane's 2 C bytes, two at a time, they took half of a token's time at K =
// 16,384: 24.3 -> 14.0 ms with the column limit for 12,000 documents).
// U > 0: for few documents at a time, the next token's first U chunks loaded
// while this one is drawn.
template <int U>
__device__ __forceinline__ void z_doc_big(const ZArgs &a, uint32_t *sm, DocRun &r, u64 *wcnt, const uint32_t *m0) {
    const int lane = threadIdx.x & 31;
    const int C = (a.K + 511) >> 9;
    const int TPL = 16 * C, PB = 512 * C;
    const uint32_t recip = static_cast<uint32_t>((0x100000000ull + TPL - 1) / TPL);     // k / TPL = umulhi(k, recip), k < 2^14
    auto pos = [=](int k) {
        const int l = static_cast<int>(__umulhi(static_cast<uint32_t>(k), recip));
        const int b = k - l * TPL;
        return ((b >> 4) << 9) + (l << 4) + (b & 15);
    };
    if (r.len == 0 || r.budget <= 0) return;
    const int planes = z_count_planes(a.narrow != 0);
    DocCounts m{reinterpret_cast<uint8_t *>(sm), PB, 0};
    build_counts(a, m, r, m0, planes, pos);
    // the topics with m > 0 as bits in topic order, in shared memory: words
    // 128 i + 4 lane to + 3 are this lane's (only it touches them)
    uint32_t *map = reinterpret_cast<uint32_t *>(m.b + planes * PB);
    int kd = 0;
    for (int w0 = 4 * lane; w0 < 16 * C; w0 += 128)
        for (int w = w0; w < w0 + 4; ++w) {
            map[w] = nonzero_topics(m, pos(32 * w), planes) | nonzero_topics(m, pos(32 * w + 16), planes) << 16;
            kd += __popc(map[w]);
        }
    kd = static_cast<int>(__reduce_add_sync(0xFFFFFFFFu, static_cast<unsigned>(kd)));
    auto flip = [&](int p) {
        const int k = ((p >> 4) & 31) * TPL + ((p >> 9) << 4) + (p & 15), w = k >> 5;
        if (((w >> 2) & 31) == lane) map[w] ^= 1u << (k & 31);
    };
    auto common = [](const uint4 x, const uint4 y) {
        return static_cast<uint32_t>(__popc(x.x & y.x) + __popc(x.y & y.y) + __popc(x.z & y.z) + __popc(x.w & y.w));
    };
    DocRun &rs = *z_warp_run(wcnt);
    if (lane == 0) rs = r;
    __syncwarp();
    uint4 *rec = token_records<0>(sm, a);
    uint32_t *drow_of = reinterpret_cast<uint32_t *>(rec + 64);
    const uint32_t sweep_end = rs.sweep + static_cast<uint32_t>(rs.max_pass_end);
    const int colmax = column_limit<0>(a.path, a.K);
    bool first = true;
    while (rs.budget > 0 && rs.sweep != sweep_end) {
        if (rs.deadline != ~0ull && !first) {
            uint64_t now = 0;
            if (lane == 0) now = global_ns();
            if (__shfl_sync(0xFFFFFFFFu, now, 0) >= rs.deadline) break;
        }
        first = false;
        const int i0 = rs.pos;
        const int cnt = static_cast<int>(min(static_cast<int64_t>(32), min(static_cast<int64_t>(rs.len - i0), rs.budget)));
        int znew = 0;
        if (lane < cnt) stage_token(a, rs, i0 + lane, rec + 2 * lane, drow_of + lane, colmax, pos);
        __syncwarp();
        uint32_t c_min = 0, c_cnt = 0, c_int = 0;      // as above, this lane's share of |J| in c_int
        uint4 ahead[U > 0 ? U : 1][3];
        auto load_ahead = [&](int tt) {
            const uint32_t dn = tt < cnt ? drow_of[tt] : 0xFFFFFFFFu;
            if (U > 0 && dn != 0xFFFFFFFFu) big_load(a.qrow + static_cast<size_t>(dn) * (3u * PB), PB, C, 0, lane, ahead);
        };
        load_ahead(0);
        for (int tt = 0; tt < cnt; ++tt) {
            const uint4 t0 = rec[2 * tt], t1 = rec[2 * tt + 1];
            TokenDraw t;
            t.kold = static_cast<int>(t1.w >> 16);
            const int n_w = static_cast<int>(t1.w & 0xFFFFu);
            t.At = (static_cast<u64>(t0.w) << 32) | t0.z;
            t.U = (static_cast<u64>(t1.x) << 32) | t1.y;
            t.ka = static_cast<int>(t0.y >> 16);
            // the next token's row on its way to L2 while this one is drawn
            if (tt + 1 < cnt) {
                const uint32_t dn = drow_of[tt + 1];
                if (dn != 0xFFFFFFFFu) {
                    const uint8_t *nrow = a.qrow + static_cast<size_t>(dn) * (3u * PB);
                    for (int o = 128 * lane; o < 3 * PB; o += 4096) asm volatile("prefetch.global.L2 [%0];" ::"l"(nrow + o));
                }
            }
            {
                const int p = t.kold;
                bool died = false;
                if (lane == ((p >> 4) & 31)) {
                    const uint32_t c = m.get(p) - 1u;
                    m.set(p, c);
                    died = c == 0;
                }
                if (__any_sync(0xFFFFFFFFu, died)) {
                    --kd;
                    flip(p);
                }
            }
            c_min += static_cast<uint32_t>(kd < n_w ? kd : n_w);
            c_cnt += kd < n_w ? 1u : 0u;
            // the word's bits, counted after the draw: nothing waits for their loads
            const uint32_t *wb = a.bits + static_cast<int64_t>(t1.z) * a.KWp;
            const uint4 early = 4 * lane < 16 * C ? *reinterpret_cast<const uint4 *>(wb + 4 * lane) : make_uint4(0u, 0u, 0u, 0u);
            const uint32_t d = drow_of[tt];
            int knew = -1;
            if (d != 0xFFFFFFFFu) {
                const uint8_t *row = a.qrow + static_cast<size_t>(d) * (3u * PB);
                u64 acc = 0;
                if constexpr (U > 0) {
                    acc = big_dot(ahead, m, PB, C, 0, lane);
                    for (int c0 = U; c0 < C; c0 += U) {
                        big_load(row, PB, C, c0, lane, ahead);
                        acc += big_dot(ahead, m, PB, C, c0, lane);
                    }
                    load_ahead(tt + 1);
                } else {
                    for (int pl = 0; pl <= m.lvl; ++pl) acc += big_plane_dot(row, m.b + pl * PB, PB, C, lane) << (8 * pl);
                }
                const u64 incl = warp_incl_scan(acc);
                u64 rb;
                knew = split_draw(t, __shfl_sync(0xFFFFFFFFu, incl, 31), rb, c_cnt);
                if (knew < 0) {
                    const int L = __ffs(__ballot_sync(0xFFFFFFFFu, rb < incl)) - 1;
                    const u64 res = __shfl_sync(0xFFFFFFFFu, rb - (incl - acc), L);
                    __syncwarp();
                    knew = big_find(L, res, row, m, PB, C, lane);
                    if (knew < 0) {
                        if (lane == 0) atomicOr(&a.stats[ST_ERROR], ERR_INTERNAL);
                        knew = t.kold;
                    }
                }
            } else {
                const int64_t col = static_cast<int64_t>((static_cast<u64>(t0.y & 0xFFFFu) << 32) | t0.x);
                load_ahead(tt + 1);
                knew = column_draw<4>(a, t, col, n_w, m, lane, c_cnt, pos);
            }
            __syncwarp();
            if (4 * lane < 16 * C) c_int += common(early, *reinterpret_cast<const uint4 *>(map + 4 * lane));
            for (int w = 128 + 4 * lane; w < 16 * C; w += 128)
                c_int += common(*reinterpret_cast<const uint4 *>(wb + w), *reinterpret_cast<const uint4 *>(map + w));
            {
                const int p = knew;
                bool born = false;
                int lv = 0;
                if (lane == ((p >> 4) & 31)) {
                    const uint32_t c = m.get(p) + 1u;
                    m.set(p, c);
                    lv = count_level(c);
                    born = c == 1;
                }
                if (__any_sync(0xFFFFFFFFu, born)) {
                    ++kd;
                    flip(p);
                }
                if (__any_sync(0xFFFFFFFFu, lv > m.lvl)) ++m.lvl;
            }
            if (lane == tt) znew = knew;
        }
        if (lane < cnt) {
            const int k = ((znew >> 4) & 31) * TPL + ((znew >> 9) << 4) + (znew & 15);
            rs.z[i0 + lane] = static_cast<int16_t>(guard_index(k, a.K, a.stats));
        }
        add_block_counts(wcnt, lane, cnt, c_min, c_cnt, c_int);
        __syncwarp();
        if (lane == 0) {
            rs.budget -= cnt;
            rs.pos += cnt;
            if (rs.pos == rs.len) { rs.pos = 0; rs.sweep += 1; }
        }
        __syncwarp();
    }
    r = rs;
    __syncwarp();
}

// NW = dense_words(K) for K <= 1024, 0 above, -1 above for few documents at a time.
template <int NW>
__device__ __forceinline__ void z_doc(const ZArgs &a, uint32_t *sm, DocRun &r, u64 *wcnt, const uint32_t *m0) {
    if constexpr (NW <= 0) z_doc_big<NW == 0 ? 0 : 8>(a, sm, r, wcnt, m0);
    else z_doc_regs<NW>(a, sm, r, wcnt, m0);
}

}  // namespace pulda
