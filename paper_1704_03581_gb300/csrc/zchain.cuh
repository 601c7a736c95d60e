// The z-step of one long document by a CTA of four warps, for the least time
// per token.
//
// A document's tokens are strictly sequential, so a long document is one
// chain of draws, and what bounds it is the instructions and latencies from
// one token's topic to the next's.  Warp 0 carries that chain and nothing
// else:
//   - warp 1 stages the tokens' records two to three blocks of 32 ahead, and
//     has the words' dense rows copied into a ring of shared-memory slots
//     (bulk copies, one group of tokens ahead), so no load on the chain goes
//     past shared memory;
//   - warp 2 replays the drawn topics one group behind, on counts of its own,
//     for the sweep's counters, and writes them out;
//   - warp 3 sums q m for token t + 1 and scans it while token t is drawn, from
//     counts (its own again) that lack token t.  The token's own weight is
//     taken off beforehand; the one thing missing, the weight of token t's new
//     topic, warp 0 adds to the scanned prefixes.  All sums are exact integers,
//     so they are those of the sequential order.
// Warp 0 finds the topic within the found lane by masked dp4a, every lane
// summing the lane's topics up to its own, without a scan.  Warps 0 and 3 meet
// once per token, all four once per group of tokens.
// About 600 cycles per token (K = 1000, a document of 3,000 tokens: 1.10 us with
// four warps sharing one token's sparse walk, 0.29 so), which warps 0 and 3 both fill: work moved from
// either to the other made a token longer (the draw's product prepared by
// warp 3 +10%, two of its scan steps left to warp 0 +5%).
// Up to kChainMaxK topics; zsplit.cuh above.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

#include "zdense.cuh"

namespace pulda {

constexpr int kChainThreads = 128;

// Tokens of a group: the ring holds three groups' rows (drawn, landed, on
// their way), within what leaves room for several CTAs per SM where rows are
// short.
__host__ __device__ __forceinline__ int chain_group(int K) {
    const int rb = dense_row_bytes(K);
    return rb <= 1536 ? 8 : rb <= 3072 ? 4 : rb <= 24576 ? 2 : 1;
}

// One token's record: {sigma_a, u}, {position of its topic | of the alias
// outcome << 16, its row's offset in shared memory or ~0, K_v, word}, {its
// column's start}.
constexpr int kChainRecWords = 12;

// Above kChainMaxK the counts of three warps and the ring no longer fit a CTA
// and zsplit.cuh takes over; the layout functions here hold for any K.
__host__ __device__ __forceinline__ int chain_count_sets(int K) { return K <= kChainMaxK ? 3 : 2; }

// Shared memory of a CTA, in bytes: the barriers and counters; the drawn
// topics of two groups; the coming token's sums; three blocks of records; the
// sets of counts (two planes each; three where a document of the launch has 2^16
// tokens or more) and, above 1024 topics, the lanes' bits; the ring.
struct CtaCtl {                 // what every kernel with a CTA per document has
    u64 full[3];                // a group's rows (zsplit.cuh: a row) have arrived
    u64 cnt[6];                 // the counters
    u64 deadline;
    int item, stop;
    int failed;                 // 1 + the barrier of a copy that did not arrive: the CTA takes no more documents
};
struct ChainCtl : CtaCtl {
    int after[2];               // after an even / odd group (a fast warp may already set the next one):
                                // kStop, kMixed: the next group holds a token without a dense row
    uint32_t drawn[16];         // two groups: position | flags
    int last[2];                // the topic of an even / odd token
    ulonglong2 ahead[2][32];    // an even / odd token's prefixes, by lane: with and without the lane's own sum
};
constexpr int kChainRecOff = 1280;
static_assert(sizeof(ChainCtl) <= kChainRecOff, "the control block must fit");
constexpr int kChainCountOff = kChainRecOff + 3 * 32 * 4 * kChainRecWords;
static_assert(kChainCountOff % 16 == 0, "counts and rows are read 16 bytes at a time");
__host__ __device__ __forceinline__ int chain_ring_off(int K, int planes = 2) {
    return kChainCountOff + planes * chain_count_sets(K) * 128 * dense_words(K) + (K > 1024 ? 16 * dense_words(K) : 0);
}
__host__ __device__ __forceinline__ int chain_smem_bytes(int K, int planes = 2) {
    return chain_ring_off(K, planes) + 3 * chain_group(K) * dense_row_bytes(K);
}
// The same for chains of any K up to kmax in one launch (shorter groups can
// take less room than the longer ones below them).
__host__ __device__ __forceinline__ int chain_smem_bytes_upto(int kmax, int planes = 2) {
    int most = 0;
    const int edge[4] = {512, 1024, kChainMaxK, kMaxK};
    for (int e : edge) {
        const int b = chain_smem_bytes(kmax < e ? kmax : e, planes);
        most = b > most ? b : most;
    }
    return most;
}
constexpr int kStop = 1, kMixed = 2;
// Flags of a drawn topic: taken from the alias table, kept for want of mass.
constexpr uint32_t kDrawnAlias = 1u << 14, kDrawnZero = 1u << 15;
static_assert(kMaxK <= (1 << 14), "positions must leave room for the flags");

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void bar_init(u64 *bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ bool bar_try_wait(u64 *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                 : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Waits for a slot, at most some seconds: false then.
__device__ __forceinline__ bool bar_wait(u64 *bar, uint32_t parity) {
    for (int i = 0; i < (1 << 22); ++i)
        if (bar_try_wait(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, uint32_t bytes, u64 *bar) {
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void bar_expect(u64 *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}

// Counts of the chain: P planes, with no test in between.
template <int P>
__device__ __forceinline__ uint32_t chain_count(const uint8_t *m, int PB, int p) {
    uint32_t c = m[p];
    if (P > 1) c |= static_cast<uint32_t>(m[p + PB]) << 8;
    if (P > 2) c |= static_cast<uint32_t>(m[p + 2 * PB]) << 16;
    return c;
}
template <int P>
__device__ __forceinline__ void chain_set(uint8_t *m, int PB, int p, uint32_t c) {
    m[p] = static_cast<uint8_t>(c);
    if (P > 1) m[p + PB] = static_cast<uint8_t>(c >> 8);
    if (P > 2) m[p + 2 * PB] = static_cast<uint8_t>(c >> 16);
}
// Whether a group of G tokens keeps counts of at most `top` in P of PL planes.
template <int P, int PL>
__device__ __forceinline__ bool chain_fits(uint32_t top, int G) {
    return P == PL || top + static_cast<uint32_t>(G) <= (P == 1 ? 255u : 65535u);
}
__device__ __forceinline__ uint32_t row_weight(const uint8_t *row, int PB, int p) {
    return row[p] | (static_cast<uint32_t>(row[p + PB]) << 8) | (static_cast<uint32_t>(row[p + 2 * PB]) << 16);
}

// What the two ranges of K do differently: NW words per lane and plane, or
// (NW = 0, K > 1024) C chunks of four.
template <int NW>
struct ChainForm {
    using G = DenseGeo<NW>;
    uint32_t mbits;             // this lane's topics with m > 0 (warp 2)
    __device__ __forceinline__ ChainForm(int) {}
    __device__ __forceinline__ static constexpr int plane() { return G::PB; }
    __device__ __forceinline__ static int pos(int k) { return G::pos(k); }
    __device__ __forceinline__ static int topic(int p) { return G::topic(p); }
    __device__ __forceinline__ static int owner(int p) { return G::owner(p); }
    __device__ __forceinline__ static uint32_t weight(const uint8_t *row, int p) { return row_weight(row, G::PB, p); }
    __device__ __forceinline__ int init_bits(const DocCounts &m, uint8_t *, int lane) {
        mbits = 0;
#pragma unroll 1
        for (int b = 0; b < G::TPL; ++b)
            if (m.get(G::lane0(b) + G::STRIDE * lane) > 0) mbits |= 1u << b;
        return __popc(mbits);
    }
    __device__ __forceinline__ void flip(int p, int lane, bool on) { mbits ^= on && lane == G::owner(p) ? 1u << G::bit(p) : 0u; }
    __device__ __forceinline__ uint32_t shared_topics(const uint32_t *bits, int lane) const {
        return static_cast<uint32_t>(__popc(lane_bits<G::TPL>(bits, 0, lane) & mbits));
    }
    template <int P>
    __device__ __forceinline__ u64 dot(const uint8_t *row, const uint8_t *m, int lane) const {
        uint32_t q[3][NW];
#pragma unroll
        for (int p = 0; p < 3; ++p) load_words<NW>(row + p * G::PB, lane, q[p]);
        u64 sum = 0;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            uint32_t w[NW];
            load_words<NW>(m + p * G::PB, lane, w);
            uint32_t s0 = 0, s1 = 0, s2 = 0;
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
    // The running sum of q m over lane L's topics up to this lane's: eight
    // lanes share two words of every plane, each summing them up to its own
    // topic (mask) with dp4a, and the groups of eight lanes before add their
    // totals.
    static constexpr int GW = NW >= 2 ? 2 : 1, GL = 4 * GW, GROUPS = NW / GW;
    __device__ __forceinline__ static void topic_masks(int lane, uint32_t (&mask)[GW]) {
        const int j = lane & (GL - 1);
#pragma unroll
        for (int x = 0; x < GW; ++x) {
            const int t = j - 4 * x;                // last topic of word x that counts
            mask[x] = t >= 3 ? 0xFFFFFFFFu : t < 0 ? 0u : (1u << (8 * (t & 3) + 8)) - 1u;
        }
    }
    template <int P>
    __device__ __forceinline__ u64 prefix(int L, const uint8_t *row, const uint8_t *m, const uint32_t (&mask)[GW], int lane) const {
        const int grp = (lane / GL) & (GROUPS - 1);
        const int at = G::lane0(GL * grp) + L * G::STRIDE;
        uint32_t q[3][GW], w[P][GW];
#pragma unroll
        for (int p = 0; p < 3; ++p) load_group(row + p * G::PB + at, q[p]);
#pragma unroll
        for (int p = 0; p < P; ++p) load_group(m + p * G::PB + at, w[p]);
        u64 sum = 0;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            uint32_t s0 = 0, s1 = 0, s2 = 0;
#pragma unroll
            for (int x = 0; x < GW; ++x) {
                s0 = __dp4a(w[p][x] & mask[x], q[0][x], s0);
                s1 = __dp4a(w[p][x] & mask[x], q[1][x], s1);
                s2 = __dp4a(w[p][x] & mask[x], q[2][x], s2);
            }
            sum += (static_cast<u64>(s0 + (s1 << 8)) + (static_cast<u64>(s2) << 16)) << (8 * p);
        }
        if constexpr (GROUPS > 1) {
            u64 t[GROUPS - 1];
#pragma unroll
            for (int g = 0; g + 1 < GROUPS; ++g) t[g] = __shfl_sync(0xFFFFFFFFu, sum, GL * g + GL - 1);
#pragma unroll
            for (int g = 0; g + 1 < GROUPS; ++g) sum += grp > g ? t[g] : 0ull;
        }
        return sum;
    }
    __device__ __forceinline__ static void load_group(const uint8_t *p, uint32_t (&w)[GW]) {
        if constexpr (GW == 2) {
            const uint2 v = *reinterpret_cast<const uint2 *>(p);
            w[0] = v.x;
            w[1] = v.y;
        } else {
            w[0] = *reinterpret_cast<const uint32_t *>(p);
        }
    }
    // lane L's topic whose running sum passes res (position, or -1)
    template <int P>
    __device__ __forceinline__ int find(int L, u64 res, const uint8_t *row, const uint8_t *m, int lane) const {
        uint32_t mask[GW];
        topic_masks(lane, mask);
        const uint32_t f = __ballot_sync(0xFFFFFFFFu, res < prefix<P>(L, row, m, mask, lane));
        return f ? G::lane0(__ffs(f) - 1) + L * G::STRIDE : -1;
    }
};
template <>
struct ChainForm<0> {
    int C, TPL, PB;
    uint32_t recip;
    uint16_t *mb;               // this lane's bits (warp 2), chunk c at mb[32 c]
    __device__ __forceinline__ ChainForm(int K) {
        C = (K + 511) >> 9;
        TPL = 16 * C;
        PB = 512 * C;
        recip = static_cast<uint32_t>((0x100000000ull + TPL - 1) / TPL);
        mb = nullptr;
    }
    __device__ __forceinline__ int plane() const { return PB; }
    __device__ __forceinline__ int pos(int k) const {
        const int l = static_cast<int>(__umulhi(static_cast<uint32_t>(k), recip));
        const int b = k - l * TPL;
        return ((b >> 4) << 9) + (l << 4) + (b & 15);
    }
    __device__ __forceinline__ int topic(int p) const { return ((p >> 4) & 31) * TPL + ((p >> 9) << 4) + (p & 15); }
    __device__ __forceinline__ static int owner(int p) { return (p >> 4) & 31; }
    __device__ __forceinline__ uint32_t weight(const uint8_t *row, int p) const { return row_weight(row, PB, p); }
    __device__ __forceinline__ int init_bits(const DocCounts &m, uint8_t *area, int lane) {
        mb = reinterpret_cast<uint16_t *>(area) + lane;
        int n = 0;
        for (int c = 0; c < C; ++c) {
            uint32_t bits = 0;
            for (int b = 0; b < 16; ++b)
                if (m.get(512 * c + 16 * lane + b) > 0) bits |= 1u << b;
            mb[32 * c] = static_cast<uint16_t>(bits);
            n += __popc(bits);
        }
        return n;
    }
    __device__ __forceinline__ void flip(int p, int lane, bool on) {
        if (on && lane == owner(p)) mb[(p >> 9) << 5] ^= static_cast<uint16_t>(1u << (p & 15));
    }
    __device__ __forceinline__ uint32_t shared_topics(const uint32_t *bits, int lane) const {
        const uint16_t *wb = reinterpret_cast<const uint16_t *>(bits) + C * lane;
        uint32_t n = 0;
        for (int c = 0; c < C; ++c) n += static_cast<uint32_t>(__popc(wb[c] & mb[32 * c]));
        return n;
    }
    template <int P>
    __device__ __forceinline__ u64 dot(const uint8_t *row, const uint8_t *m, int lane) const {
        u64 sum = big_plane_dot(row, m, PB, C, lane);
        if (P > 1) sum += big_plane_dot(row, m + PB, PB, C, lane) << 8;
        if (P > 2) sum += big_plane_dot(row, m + 2 * PB, PB, C, lane) << 16;
        return sum;
    }
    template <int P>
    __device__ __forceinline__ int find(int L, u64 res, const uint8_t *row, uint8_t *m, int lane) const {
        return big_find(L, res, row, DocCounts{m, PB, P - 1}, PB, C, lane);
    }
};

__device__ __forceinline__ void pair_barrier() { asm volatile("bar.sync 1, 64;" ::: "memory"); }     // warps 0 and 3

// What warps 0 and 3 each carry from token to token.
struct ChainState {
    int prev;                   // the last token's new topic, not in the counts yet (at a document's
                                // start the first token's topic, taken out of the counts)
    uint32_t top;               // a bound on every count
    uint32_t bad;               // a draw found no topic
};

// The last token's topic into the counts, this one's out.  Every lane stores
// the same bytes, once every lane has read the old ones.
template <int P>
__device__ __forceinline__ void chain_update(uint8_t *m, int PB, int kold, ChainState &st) {
    const uint32_t c1 = chain_count<P>(m, PB, st.prev) + 1u;
    const uint32_t c0 = (st.prev == kold ? c1 : chain_count<P>(m, PB, kold)) - 1u;
    __syncwarp();
    chain_set<P>(m, PB, st.prev, c1);
    chain_set<P>(m, PB, kold, c0);
    st.top = max(st.top, c1);
}

// The lanes' sums, in the counts at hand, for the token of record part r1, less
// the token itself; prefixes with and without the lane's own.
template <int NW, int P>
__device__ __forceinline__ ulonglong2 chain_sums(const ChainForm<NW> &form, const uint8_t *sm, const uint8_t *m, const uint4 r1, int lane) {
    const u64 sum = form.template dot<P>(sm + r1.y, m, lane) - (lane == form.owner(static_cast<int>(r1.x & 0xFFFFu)) ? r1.z : 0u);
    const u64 incl = warp_incl_scan<32>(sum);
    return make_ulonglong2(incl, incl - sum);
}

// Where a pass stands: n tokens in ng groups of G, group g next.
struct ChainPass {
    int n, ng, G, g;
    int done;                   // tokens drawn
    int after;                  // what warp 1 said after the last group
    __device__ __forceinline__ int group_tokens() const { return min(G, n - g * G); }
    // the end of a group: all four warps
    __device__ __forceinline__ void meet(const ChainCtl &ctl) {
        done += group_tokens();
        __syncthreads();
        after = ctl.after[g & 1];
        ++g;
    }
    __device__ __forceinline__ bool more() const { return g < ng && !(after & kStop); }
};

// Warp 3: the sums of the token after each of the coming groups' tokens, while
// that one is drawn; for as long as counts stay in P planes.
template <int NW, int P, int PL>
__device__ __forceinline__ void chain_run_ahead(const ChainForm<NW> &form, uint8_t *sm, ChainCtl &ctl, uint8_t *m, ChainPass &ps,
                                                ChainState &st) {
    const int lane = threadIdx.x & 31;
    const int PB = form.plane();
    const uint4 *recs = reinterpret_cast<const uint4 *>(sm + kChainRecOff), *end = recs + 3 * 96;
    int t = ps.g * ps.G;
    const uint4 *rec = recs + 3 * (t % 96);
    uint4 r1 = rec[1];
    do {
        const int cnt = ps.group_tokens();
#pragma unroll 1
        for (int u = 0; u < cnt; ++u, ++t) {
            const int kold = static_cast<int>(r1.x & 0xFFFFu);
            rec = rec + 3 == end ? recs : rec + 3;
            const uint4 n1 = rec[1];
            if (st.prev < 0) st.prev = ctl.last[(t + 1) & 1];           // token t - 1's, drawn meanwhile
            if (n1.y != 0xFFFFFFFFu) {
                // from the counts as they were, less this token's and its own
                // topic (nothing here waits for a draw); then with the new
                // topic of the token before, in the prefixes
                const uint8_t *row = sm + n1.y;
                const u64 sum = form.template dot<P>(row, m, lane) - (lane == form.owner(kold) ? n1.w : 0u) -
                                (lane == form.owner(static_cast<int>(n1.x & 0xFFFFu)) ? n1.z : 0u);
                const uint32_t dn = form.weight(row, st.prev);
                const int ow = form.owner(st.prev);
                const u64 incl = warp_incl_scan<32>(sum);
                ctl.ahead[(t + 1) & 1][lane] = make_ulonglong2(incl + (lane >= ow ? dn : 0u), incl - sum + (lane > ow ? dn : 0u));
            }
            chain_update<P>(m, PB, kold, st);
            st.prev = -1;
            r1 = n1;
            pair_barrier();
        }
        ps.meet(ctl);
    } while (ps.more() && chain_fits<P, PL>(st.top, ps.G));
}

// Warp 0: the coming groups, while every token of theirs has a dense row and
// counts stay in P planes.
template <int NW, int P, int PL>
__device__ __forceinline__ void chain_run_fast(const ChainForm<NW> &form, uint8_t *sm, ChainCtl &ctl, uint8_t *m, ChainPass &ps,
                                               ChainState &st) {
    using G = DenseGeo<NW>;
    const int lane = threadIdx.x & 31;
    uint32_t mask[ChainForm<NW>::GW];
    form.topic_masks(lane, mask);
    const uint4 *recs = reinterpret_cast<const uint4 *>(sm + kChainRecOff), *end = recs + 3 * 96;
    int t = ps.g * ps.G;
    const uint4 *rec = recs + 3 * (t % 96);
    uint4 r1 = rec[1];
    uint32_t delta = form.weight(sm + r1.y, st.prev);
    do {
        const int cnt = ps.group_tokens();
        uint32_t *drawn = ctl.drawn + 8 * (ps.g & 1);
#pragma unroll 1
        for (int u = 0; u < cnt; ++u, ++t) {
            const uint4 r0 = rec[0];
            rec = rec + 3 == end ? recs : rec + 3;
            const uint4 n1 = rec[1];
            const uint8_t *row = sm + r1.y, *nrow = sm + (n1.y == 0xFFFFFFFFu ? r1.y : n1.y);
            const u64 At = (static_cast<u64>(r0.y) << 32) | r0.x, U = (static_cast<u64>(r0.w) << 32) | r0.z;
            const int kold = static_cast<int>(r1.x & 0xFFFFu);
            const ulonglong2 mine = ctl.ahead[t & 1][lane];
            const u64 all = ctl.ahead[t & 1][31].x;
            const int ow = G::owner(st.prev);
            chain_update<P>(m, G::PB, kold, st);
            const u64 upto = mine.x + (lane >= ow ? delta : 0u), below = mine.y + (lane > ow ? delta : 0u);
            const u64 T = At + ((all + delta) << kFracBits);
            const u64 rr = __umul64hi(U, T);
            const u64 rb = (rr - At) >> kFracBits;
            // no lane passes for an alias draw (rr < At wraps round) or without any
            // mass: the outcome then does not wait for the rest
            const uint32_t bal = __ballot_sync(0xFFFFFFFFu, rb < upto);
            const uint32_t other = rr < At ? (r1.x >> 16) | kDrawnAlias : static_cast<uint32_t>(kold) | kDrawnZero;
            const int L = (__ffs(bal) - 1) & 31;
            const u64 res = __shfl_sync(0xFFFFFFFFu, rb - below, L);
            const uint32_t f = __ballot_sync(0xFFFFFFFFu, res < form.template prefix<P>(L, row, m, mask, lane));
            const uint32_t knew = bal ? static_cast<uint32_t>(G::lane0((__ffs(f) - 1) & 31) + L * G::STRIDE) : other;
            st.prev = static_cast<int>(knew & 0x3FFFu);
            ctl.last[t & 1] = st.prev;
            delta = form.weight(nrow, st.prev);         // the next token's, on its way over the barrier
            drawn[u] = knew;
            st.bad |= bal != 0 && f == 0 ? 1u : 0u;
            r1 = n1;
            pair_barrier();
        }
        ps.meet(ctl);
    } while (ps.more() && !(ps.after & kMixed) && chain_fits<P, PL>(st.top, ps.G));
}

// The same for any group: tokens without a dense row among them, or K > 1024.
template <int NW, int P>
__device__ __forceinline__ void chain_group_any(const ZArgs &a, const ChainForm<NW> &form, uint8_t *sm, ChainCtl &ctl, uint8_t *m, int t,
                                                int cnt, uint32_t *drawn, ChainState &st) {
    const int lane = threadIdx.x & 31;
    const int PB = form.plane();
    const uint4 *recs = reinterpret_cast<const uint4 *>(sm + kChainRecOff);
#pragma unroll 1
    for (int u = 0; u < cnt; ++u, ++t) {
        const uint4 *rec = recs + 3 * (t % 96);
        const uint4 r0 = rec[0], r1 = rec[1];
        const u64 At = (static_cast<u64>(r0.y) << 32) | r0.x, U = (static_cast<u64>(r0.w) << 32) | r0.z;
        const int kold = static_cast<int>(r1.x & 0xFFFFu);
        const bool dense = r1.y != 0xFFFFFFFFu;
        const uint8_t *row = sm + r1.y;
        const uint32_t delta = dense ? form.weight(row, st.prev) : 0u;
        const int ow = form.owner(st.prev);
        const ulonglong2 mine = ctl.ahead[t & 1][lane];
        chain_update<P>(m, PB, kold, st);
        __syncwarp();
        const u64 upto = mine.x + (lane >= ow ? delta : 0u), below = mine.y + (lane > ow ? delta : 0u);
        uint32_t knew;
        if (dense) {
            const u64 rr = __umul64hi(U, At + (__shfl_sync(0xFFFFFFFFu, upto, 31) << kFracBits));
            if (rr < At) {
                knew = (r1.x >> 16) | kDrawnAlias;
            } else {
                const u64 rb = (rr - At) >> kFracBits;
                const uint32_t bal = __ballot_sync(0xFFFFFFFFu, rb < upto);
                knew = static_cast<uint32_t>(kold) | kDrawnZero;
                if (bal) {
                    const int L = __ffs(bal) - 1;
                    const u64 res = __shfl_sync(0xFFFFFFFFu, rb - below, L);
                    const int k = form.template find<P>(L, res, row, m, lane);
                    st.bad |= k < 0 ? 1u : 0u;
                    knew = static_cast<uint32_t>(k < 0 ? kold : k);
                }
            }
        } else {
            const uint4 r2 = rec[2];
            uint32_t c = 0;
            DocCounts mc{m, PB, P - 1};
            const TokenDraw td{At, U, static_cast<int>(r1.x >> 16), kold};
            const int k = column_draw<4>(a, td, static_cast<int64_t>((static_cast<u64>(r2.y) << 32) | r2.x), static_cast<int>(r2.z), mc, lane, c,
                                      [&](int x) { return form.pos(x); });
            knew = static_cast<uint32_t>(k) | (c & (1u << 6) ? kDrawnAlias : 0u) | (c & (1u << 12) ? kDrawnZero : 0u);
        }
        drawn[u] = knew;
        st.prev = static_cast<int>(knew & 0x3FFFu);
        ctl.last[t & 1] = st.prev;
        pair_barrier();
        __syncwarp();
    }
}

// A run's topics counted by every thread of the CTA, K 32-bit counts in `hist`:
// shared memory that bulk copies write later, behind async_reuse() and a barrier.
// Warps that each count the tokens for themselves wait on one load per 32: 1 us
// of them, so 3 ms for 90,000 tokens, in every launch of a request that long (us
// per token of 66,000, K = 1,000: 0.312 -> 0.297).  The counts' way through K
// words costs more where documents are short (K = 3,000, 200 tokens 0.742 ->
// 0.758, 1,000 0.662 -> 0.656; K = 8,000, 600 tokens 0.874 -> 0.889).
__device__ __forceinline__ int chain_hist_tokens(int K) { return 128 + K / 8; }
constexpr int kCtaHistBatch = 8;
__device__ __forceinline__ void cta_histogram(const ZArgs &a, const DocRun &r, uint32_t *hist) {
    for (int k = threadIdx.x; k < a.K; k += blockDim.x) hist[k] = 0;
    __syncthreads();
    const int T = blockDim.x;
    int i = threadIdx.x;
    for (; i + (kCtaHistBatch - 1) * T < r.len; i += kCtaHistBatch * T) {
        int k[kCtaHistBatch];
#pragma unroll
        for (int u = 0; u < kCtaHistBatch; ++u) k[u] = r.z[i + u * T];
#pragma unroll
        for (int u = 0; u < kCtaHistBatch; ++u) atomicAdd(&hist[guard_index(k[u], a.K, a.stats)], 1u);
    }
    for (; i < r.len; i += T) atomicAdd(&hist[guard_index(r.z[i], a.K, a.stats)], 1u);
    __syncthreads();
}
__device__ __forceinline__ void async_reuse() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// One warp's counts from them: PL planes, and lvl.
template <int PL, typename Pos>
__device__ __forceinline__ void counts_from(const uint32_t *hist, int K, DocCounts &m, Pos pos) {
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < PL * m.PB / 16; i += 32) reinterpret_cast<uint4 *>(m.b)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    int top = 0;
    for (int k = lane; k < K; k += 32) {
        const uint32_t c = hist[k];
        if (c) chain_set<PL>(m.b, m.PB, pos(k), c);
        top = max(top, count_level(c));
    }
    m.lvl = static_cast<int>(__reduce_max_sync(0xFFFFFFFFu, static_cast<unsigned>(top)));
    __syncwarp();
}

// A copy did not arrive in time (one warp): the error, and the CTA gives up, but
// not before the copy, if it comes.
__device__ __forceinline__ void cta_failed(const ZArgs &a, CtaCtl &ctl, uint32_t phases) {
    if ((threadIdx.x & 31) == 0) atomicOr(&a.stats[ST_ERROR], ERR_COPY);
    const int s = ctl.failed - 1;
    bar_wait(&ctl.full[s], (phases >> s) & 1u);
}

// All threads of the CTA; sm: chain_smem_bytes(K) bytes.  phases: the parities
// of the groups' barriers, kept from one document to the next.  PL planes of
// counts: two for documents of at most kNarrowMaxLen tokens, three for any.
template <int NW, int PL>
__device__ __forceinline__ void z_doc_chain(const ZArgs &a, uint8_t *sm, DocRun &r, uint32_t &phases) {
    const int lane = threadIdx.x & 31;
    const int role = threadIdx.x >> 5;      // 0: the chain, 1: records and rows, 2: counters and topics, 3: sums ahead
    const int K = a.K;
    if (r.len == 0 || r.budget <= 0) return;
    ChainCtl &ctl = *reinterpret_cast<ChainCtl *>(sm);
    uint4 *recs = reinterpret_cast<uint4 *>(sm + kChainRecOff);
    const int ring = chain_ring_off(K, PL), RB = dense_row_bytes(K), G = chain_group(K);
    ChainForm<NW> form(K);
    const int PB = form.plane();
    auto pos = [&](int k) { return form.pos(k); };
    // warps 0, 2 and 3 each keep the document's counts
    DocCounts m{sm + kChainCountOff + (role == 0 ? 0 : role == 2 ? PL * PB : 2 * PL * PB), PB, 0};
    if (r.len >= chain_hist_tokens(K)) {
        uint32_t *hist = reinterpret_cast<uint32_t *>(sm + ring);
        cta_histogram(a, r, hist);
        if (role != 1) counts_from<PL>(hist, K, m, pos);
        async_reuse();
    } else if (role != 1) {
        build_counts(a, m, r, nullptr, PL, pos);
    }
    ChainState st{};
    st.prev = -1;
    bool begun = false;
    int kd = 0;
    if (role == 0 || role == 3) {
        uint32_t top = 0;
        for (int p = lane; p < PB; p += 32) top = max(top, chain_count<PL>(m.b, PB, p));
        st.top = __reduce_max_sync(0xFFFFFFFFu, top);
    } else if (role == 2) {
        kd = static_cast<int>(__reduce_add_sync(0xFFFFFFFFu, static_cast<unsigned>(form.init_bits(m, sm + kChainCountOff + PL * chain_count_sets(K) * PB, lane))));
    }
    constexpr int colmax = -1;     // a row wherever there is one
    const uint32_t sweep_end = r.sweep + static_cast<uint32_t>(r.max_pass_end);
    bool stop = false;
    while (!stop && r.budget > 0 && r.sweep != sweep_end) {
        // one pass, or what of it the budget allows: n tokens from r.pos
        const int p0 = r.pos;
        const int n = static_cast<int>(min(static_cast<int64_t>(r.len - p0), r.budget));
        const int ng = (n + G - 1) / G;
        StagedToken tok;
        auto record = [&](int t) {
            uint4 *rec = recs + 3 * (t % 96);
            if (t == n) rec[1] = make_uint4(0u, static_cast<uint32_t>(ring), 0u, 0u);     // the stand-in after the last token
            if (t >= n) return;
            const uint32_t ka = static_cast<uint32_t>(pos(tok.load_alias(a)));
            rec[0] = make_uint4(static_cast<uint32_t>(tok.A), static_cast<uint32_t>(tok.A >> 32), tok.x.y, tok.x.x);
            rec[1] = make_uint4(static_cast<uint32_t>(pos(tok.topic)) | (ka << 16),
                                tok.row == 0xFFFFFFFFu ? tok.row : static_cast<uint32_t>(ring + (t % (3 * G)) * RB), 0u, tok.row);
            rec[2] = make_uint4(static_cast<uint32_t>(tok.col), static_cast<uint32_t>(static_cast<u64>(tok.col) >> 32),
                                static_cast<uint32_t>(tok.n_w), static_cast<uint32_t>(tok.word));
        };
        // block b, a step at a time (lane l its token l)
        auto stage = [&](int b, int step) {
            const int t = 32 * b + lane;
            if (step == 0 && t < n) tok.load_token(a, r, p0 + t);
            if (step == 1 && t < n) tok.load_word(a, colmax);
            if (step == 2) record(t);
        };
        // group g's rows on their way (lane u < G its token u)
        auto fetch = [&](int g) {
            const int t = g * G + lane;
            uint32_t at = 0xFFFFFFFFu, d = 0;
            if (lane < G && t < n) {
                at = recs[3 * (t % 96) + 1].y;
                d = recs[3 * (t % 96) + 1].w;
            }
            const int rows = __popc(__ballot_sync(0xFFFFFFFFu, at != 0xFFFFFFFFu));
            u64 *bar = &ctl.full[g % 3];
            if (lane == 0) bar_expect(bar, static_cast<uint32_t>(rows * RB));
            __syncwarp();
            if (at != 0xFFFFFFFFu) bulk_copy(sm + at, a.qrow + static_cast<size_t>(d) * RB, static_cast<uint32_t>(RB), bar);
        };
        auto landed = [&](int g) {
            const int s = g % 3;
            const bool ok = bar_wait(&ctl.full[s], (phases >> s) & 1u);
            if (ok) phases ^= 1u << s;
            else if (lane == 0) ctl.failed = 1 + s;
            // the weights of the tokens' own and previous topics, now that their rows are here
            const int t = g * G + lane;
            if (ok && lane < G && t < n) {
                uint4 *r1 = recs + 3 * (t % 96) + 1;
                if (r1->y != 0xFFFFFFFFu) {
                    r1->z = form.weight(sm + r1->y, static_cast<int>(r1->x & 0xFFFFu));
                    if (t > 0) r1->w = form.weight(sm + r1->y, static_cast<int>(recs[3 * ((t - 1) % 96) + 1].x & 0xFFFFu));
                }
            }
            __syncwarp();
            return ok;
        };
        // whether group g holds a token without a row
        auto mixed = [&](int g) {
            const int t = g * G + lane;
            return __any_sync(0xFFFFFFFFu, lane < G && t < n && recs[3 * (t % 96) + 1].y == 0xFFFFFFFFu) != 0;
        };
        // the counters and topics of group g, as drawn
        auto replay = [&](int g) {
            const int t0 = g * G, cnt = min(G, n - t0);
            constexpr int GM = NW == 0 ? 1 : NW == 8 ? 4 : 8;       // chain_group(K), K <= 1024
            uint32_t wb[GM];
            if constexpr (NW > 0) {
#pragma unroll
                for (int u = 0; u < GM; ++u)
                    if (u < cnt) wb[u] = lane_bits<DenseGeo<NW>::TPL>(a.bits, static_cast<int64_t>(recs[3 * ((t0 + u) % 96) + 2].w) * a.KWp, lane);
            }
            uint32_t c_min = 0, c_cnt = 0, c_int = 0;
            auto token = [&](int u, uint32_t bits) {
                const int kold = static_cast<int>(recs[3 * ((t0 + u) % 96) + 1].x & 0xFFFFu);
                const uint4 r2 = recs[3 * ((t0 + u) % 96) + 2];
                const uint32_t x = ctl.drawn[8 * (g & 1) + u];
                const int knew = static_cast<int>(x & 0x3FFFu), n_w = static_cast<int>(r2.z);
                const uint32_t co = chain_count<PL>(m.b, PB, kold) - 1u;
                __syncwarp();
                chain_set<PL>(m.b, PB, kold, co);
                if (co == 0) --kd;
                form.flip(kold, lane, co == 0);
                c_min += static_cast<uint32_t>(kd < n_w ? kd : n_w);
                c_cnt += (kd < n_w ? 1u : 0u) + (x & kDrawnAlias ? 1u << 6 : 0u) + (x & kDrawnZero ? 1u << 12 : 0u);
                if constexpr (NW > 0) c_int += static_cast<uint32_t>(__popc(bits & form.mbits));
                else c_int += form.shared_topics(a.bits + static_cast<int64_t>(r2.w) * a.KWp, lane);
                const uint32_t cn = chain_count<PL>(m.b, PB, knew) + 1u;
                __syncwarp();
                chain_set<PL>(m.b, PB, knew, cn);
                if (cn == 1) ++kd;
                form.flip(knew, lane, cn == 1);
            };
            if constexpr (NW > 0) {
#pragma unroll
                for (int u = 0; u < GM; ++u)
                    if (u < cnt) token(u, wb[u]);
            } else {
                for (int u = 0; u < cnt; ++u) token(u, 0u);
            }
            if (lane < cnt) {
                const int k = form.topic(static_cast<int>(ctl.drawn[8 * (g & 1) + lane] & 0x3FFFu));
                r.z[p0 + t0 + lane] = static_cast<int16_t>(guard_index(k, K, a.stats));
            }
            add_block_counts(ctl.cnt, lane, cnt, c_min, c_cnt, c_int);
        };
        __syncthreads();            // the last pass's topics are written and its records done with
        if (role < 3)
            for (int step = 0; step < 3; ++step) stage(role, step);
        __syncthreads();
        bool ok = true;
        if (role == 1) {
            fetch(0);
            if (ng > 1) fetch(1);
            ok = landed(0);
            if (ng > 1) ok = landed(1) && ok;
            const bool mix = mixed(0);
            if (lane == 0) ctl.stop = (ok ? 0 : kStop) | (mix ? kMixed : 0);
        }
        __syncthreads();
        ChainPass ps{n, ng, G, 0, 0, ctl.stop};
        if ((role == 0 || role == 3) && ps.more()) {
            const uint4 r1 = recs[1];
            if (!begun) {
                st.prev = static_cast<int>(r1.x & 0xFFFFu);
                const uint32_t c = chain_count<PL>(m.b, PB, st.prev) - 1u;
                __syncwarp();
                chain_set<PL>(m.b, PB, st.prev, c);
                __syncwarp();
            }
            if (r1.y != 0xFFFFFFFFu && role == 3) ctl.ahead[0][lane] = chain_sums<NW, PL>(form, sm, m.b, r1, lane);
            begun = true;
        }
        __syncthreads();
        while (ps.more()) {
            const int g = ps.g, t0 = g * G, cnt = ps.group_tokens();
            // counts stay in one plane, or two
            const bool one = chain_fits<1, PL>(st.top, G), two = chain_fits<2, PL>(st.top, G);
            if (role == 0) {
                uint32_t *drawn = ctl.drawn + 8 * (g & 1);
                if constexpr (NW > 0) {
                    if (!(ps.after & kMixed)) {
                        if (one) chain_run_fast<NW, 1, PL>(form, sm, ctl, m.b, ps, st);
                        else if (two) chain_run_fast<NW, 2, PL>(form, sm, ctl, m.b, ps, st);
                        else chain_run_fast<NW, PL, PL>(form, sm, ctl, m.b, ps, st);
                        continue;
                    }
                    chain_group_any<NW, PL>(a, form, sm, ctl, m.b, t0, cnt, drawn, st);
                } else {
                    if (one) chain_group_any<NW, 1>(a, form, sm, ctl, m.b, t0, cnt, drawn, st);
                    else if (two) chain_group_any<NW, 2>(a, form, sm, ctl, m.b, t0, cnt, drawn, st);
                    else chain_group_any<NW, PL>(a, form, sm, ctl, m.b, t0, cnt, drawn, st);
                }
            } else if (role == 3) {
                if (one) chain_run_ahead<NW, 1, PL>(form, sm, ctl, m.b, ps, st);
                else if (two) chain_run_ahead<NW, 2, PL>(form, sm, ctl, m.b, ps, st);
                else chain_run_ahead<NW, PL, PL>(form, sm, ctl, m.b, ps, st);
                continue;
            } else if (role == 1) {
                if (g + 2 < ng) fetch(g + 2);
                // block b - 1 was drawn before this block's second group, and is
                // replayed then: block b + 2 takes its place, a step a group, so
                // that no step's loads are waited for
                const int b = t0 >> 5, step = (t0 & 31) / G - 1;
                if (b > 0 && 32 * (b + 2) <= n) {
                    if (step >= 0 && step < 3) stage(b + 2, step);
                    __syncwarp();
                }
                if (g + 2 < ng) ok = landed(g + 2);
                // the deadline, after every block of 32 and every pass (a document may be shorter than a block)
                const bool late = (((t0 + cnt) & 31) == 0 || g + 1 == ng) && r.deadline != ~0ull && global_ns() >= r.deadline;
                const bool mix = g + 1 < ng && mixed(g + 1);
                if (lane == 0) ctl.after[g & 1] = (late || !ok ? kStop : 0) | (mix ? kMixed : 0);
            } else if (g > 0) {
                replay(g - 1);
            }
            ps.meet(ctl);
        }
        const int done = ps.done;
        stop = (ps.after & kStop) != 0;
        if (role == 2 && done > 0) replay((done - 1) / G);
        if (role == 3 && done > 0) st.prev = ctl.last[(done - 1) & 1];
        if (role == 0 && lane == 0 && st.bad) atomicOr(&a.stats[ST_ERROR], ERR_INTERNAL);
        r.budget -= done;
        r.pos += done;
        if (r.pos == r.len) { r.pos = 0; r.sweep += 1; }
    }
    __syncthreads();
    if (role == 1 && ctl.failed) cta_failed(a, ctl, phases);
}

// Before the first document: the groups' barriers and the counters.
__device__ __forceinline__ void cta_begin(uint8_t *sm) {
    CtaCtl &ctl = *reinterpret_cast<CtaCtl *>(sm);
    if (threadIdx.x == 0) {
        for (int s = 0; s < 3; ++s) bar_init(&ctl.full[s]);
        for (int s = 0; s < 6; ++s) ctl.cnt[s] = 0;
        ctl.stop = ctl.failed = 0;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
}

}  // namespace pulda
