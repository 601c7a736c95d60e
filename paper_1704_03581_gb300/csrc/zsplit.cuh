// The z-step of one document by a CTA above 8,192 topics: four warps on each
// token, and two that serve them.
//
// There the chain of zchain.cuh has no room for the sums ahead (a row is 25 to
// 48 KB), and one warp over a whole row is what bounds a token.  Here warp w of
// the four takes the w-th quarter of every lane's chunks: it keeps those
// topics' counts up to date, sums q m over them, and looks for the draw among
// them when it falls there, so no byte of the counts is written by one warp and
// read by another but where a barrier lies between.  Two barriers per token:
//   - every thread stores its sum, the last token's topic in its counts first;
//   - A: every warp scans the 128 sums and draws; the warp of the sum that
//     passes the draw finds the topic, and the next token's own topic goes out
//     of the counts;
//   - B: every thread reads it.
// A word of up to kSplitColumn topics is summed over its column instead, four
// entries per thread; a longer column only where the word has no row.  The
// fifth warp stages the tokens' records, has the rows copied into a ring of
// three, two tokens ahead, and one token behind keeps the sweep's counters and
// writes the topics out; the sixth brings the next token's short column.
// Documents of any length: three count planes.
// What bounds it: the 1,800 to 2,400 cycles from one token's topic to the
// next's, most of them instruction latencies with a warp or two per scheduler.
// One document of 3,000 tokens, us per token at K = 8,200 / 12,000 / 16,384,
// columns of 300 topics on average: one warp over rows 1.51 / 2.47 / 2.02, four
// warps over columns as they lie in memory 0.97 / 1.01 / 1.03, this 0.97 / 1.05 /
// 1.06; columns of 4,100 / 5,600 / 7,200 topics: 1.45 / 1.69 / 1.97, 4.2 / 5.0 /
// 6.8, and 1.19 / 1.22 / 1.26.  The column limit: 256 takes 1.04 and 1.15 us at
// the short columns of K = 8,200 and 16,384, 384 1.01 and 1.07, 512 0.94 and
// 1.05; entries past 512, eight per thread, gained nothing.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

#include "zchain.cuh"

namespace pulda {

constexpr int kSplitWarps = 4;                      // that draw
constexpr int kSplitThreads = 32 * (kSplitWarps + 2);
constexpr int kSplitEntries = 4;                    // of a short column, per thread
constexpr int kSplitColumn = kSplitEntries * 32 * kSplitWarps;
constexpr int kSplitMapWords = kMaxK / 32;          // of the document's topics as bits

// A CTA's shared memory: the control block, the bits, two short columns, two
// blocks of 32 records, three count planes, three rows.  Pairs are of even / odd
// tokens, fours of token t at t & 3.
struct SplitCtl : CtaCtl {
    int kd;
    int bad[2], halt[2];        // the next token's row did not arrive; the deadline has passed
    int high;                   // the highest plane some count has reached
    int drawn[2];               // the token's position | flags (kDrawnAlias, kDrawnZero)
    int born[4], died[4];       // the last token's topic is new to the document, this token's own was its last
    alignas(16) u64 part[32 * kSplitWarps];     // the threads' sums, in topic order
};
constexpr int kSplitMapOff = (sizeof(SplitCtl) + 15) / 16 * 16;
constexpr int kSplitColOff = kSplitMapOff + 4 * kSplitMapWords;
constexpr int kSplitColBytes = kSplitColumn * (4 + 2);      // q, then positions
constexpr int kSplitRecOff = kSplitColOff + 2 * kSplitColBytes;
constexpr int kSplitCountOff = kSplitRecOff + 2 * 4 * 32 * kTokRecWords;
static_assert(kSplitColOff % 16 == 0 && kSplitColBytes % 16 == 0 && kSplitRecOff % 16 == 0 && kSplitCountOff % 16 == 0, "counts and rows are read 16 bytes at a time");
__host__ __device__ __forceinline__ int split_smem_bytes(int K) { return kSplitCountOff + 4 * dense_row_bytes(K); }

__device__ __forceinline__ void split_barrier() { asm volatile("bar.sync 1, 128;" ::: "memory"); }     // the four warps

__device__ __forceinline__ void z_doc_split(const ZArgs &a, uint8_t *sm, DocRun &r, uint32_t &phases) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool service = warp >= kSplitWarps;
    const int K = a.K;
    if (r.len == 0 || r.budget <= 0) return;
    SplitCtl &x = *reinterpret_cast<SplitCtl *>(sm);
    uint32_t *map = reinterpret_cast<uint32_t *>(sm + kSplitMapOff);
    const ChainForm<0> form(K);
    const int C = form.C, PB = form.PB, RB = 3 * PB;
    uint8_t *counts = sm + kSplitCountOff, *ring = counts + 3 * PB;
    auto pos = [&](int k) { return form.pos(k); };
    auto rec_of = [&](int t) { return reinterpret_cast<uint4 *>(sm + kSplitRecOff) + 2 * (t & 63); };
    auto row_of = [&](int t) { return reinterpret_cast<uint32_t *>(sm + kSplitRecOff + 64 * 32) + (t & 63); };
    auto col_of = [&](int t) { return sm + kSplitColOff + (t & 1) * kSplitColBytes; };
    const int planes = r.len <= kNarrowMaxLen ? 2 : 3;
    DocCounts all{counts, PB, planes - 1};
    for (int i = threadIdx.x; i < planes * PB / 16; i += kSplitThreads) reinterpret_cast<uint4 *>(counts)[i] = make_uint4(0u, 0u, 0u, 0u);
    uint32_t *hist = reinterpret_cast<uint32_t *>(ring);
    cta_histogram(a, r, hist);
    for (int k = threadIdx.x; k < K; k += kSplitThreads)
        if (hist[k]) all.set(pos(k), hist[k]);
    async_reuse();
    if (threadIdx.x == 0) x.kd = x.high = x.bad[0] = x.bad[1] = 0;
    __syncthreads();
    // this thread's topics: lane `lane`'s chunks [c0, c1), and the planes they take
    const int per = (C + kSplitWarps - 1) / kSplitWarps, c0 = min(C, warp * per), c1 = min(C, c0 + per);
    auto mine = [&](int p) { return ((p >> 4) & 31) == lane && static_cast<unsigned>((p >> 9) - c0) < static_cast<unsigned>(c1 - c0); };
    DocCounts m{counts, PB, 0};
    for (int pl = 1; pl < planes; ++pl)
        for (int c = c0; c < c1; ++c) {
            const uint4 v = *reinterpret_cast<const uint4 *>(counts + pl * PB + 512 * c + 16 * lane);
            if (v.x | v.y | v.z | v.w) m.lvl = pl;
        }
    if (m.lvl > 0) atomicMax(&x.high, m.lvl);
    // the document's topics as bits, in topic order
    for (int w = threadIdx.x; w < kSplitMapWords; w += kSplitThreads) {
        const uint32_t bits = w < 16 * C ? nonzero_topics(all, pos(32 * w), planes) | nonzero_topics(all, pos(32 * w + 16), planes) << 16 : 0u;
        map[w] = bits;
        if (bits) atomicAdd(&x.kd, __popc(bits));
    }
    __syncthreads();
    int kd = x.kd;
    int prev = -1;              // the last token's new topic
    int due = -1;               // the same while it is not in the counts (the four warps)
    const uint32_t sweep_end = r.sweep + static_cast<uint32_t>(r.max_pass_end);
    bool stop = false, ok = true;
    while (!stop && r.budget > 0 && r.sweep != sweep_end) {
        // one pass, or what of it the budget allows: n tokens from r.pos
        const int p0 = r.pos;
        const int n = static_cast<int>(min(static_cast<int64_t>(r.len - p0), r.budget));
        StagedToken tok;
        // block b, a step at a time (lane l its token l)
        auto stage = [&](int b, int step) {
            const int t = 32 * b + lane;
            if (t >= n) return;
            if (step == 0) tok.load_token(a, r, p0 + t);
            if (step == 1) tok.load_word(a, kSplitColumn);
            if (step == 2) {
                const uint32_t ka = static_cast<uint32_t>(pos(tok.load_alias(a)));
                uint4 *rec = rec_of(t);
                rec[0] = make_uint4(static_cast<uint32_t>(tok.col), static_cast<uint32_t>(static_cast<u64>(tok.col) >> 32) | (ka << 16),
                                    static_cast<uint32_t>(tok.A), static_cast<uint32_t>(tok.A >> 32));
                rec[1] = make_uint4(tok.x.x, tok.x.y, static_cast<uint32_t>(tok.word),
                                    static_cast<uint32_t>(tok.n_w) | (static_cast<uint32_t>(pos(tok.topic)) << 16));
                *row_of(t) = tok.row;
            }
        };
        // token t's row on its way into slot t % 3 (one thread)
        auto fetch = [&](int t) {
            const uint32_t d = t < n ? *row_of(t) : 0xFFFFFFFFu;
            if (d == 0xFFFFFFFFu) return;
            u64 *bar = &x.full[t % 3];
            bar_expect(bar, static_cast<uint32_t>(RB));
            bulk_copy(ring + (t % 3) * RB, a.qrow + static_cast<size_t>(d) * RB, static_cast<uint32_t>(RB), bar);
        };
        auto landed = [&](int t) {
            if (t >= n || *row_of(t) == 0xFFFFFFFFu) return true;
            const int s = t % 3;
            const bool here = bar_wait(&x.full[s], (phases >> s) & 1u);
            if (here) phases ^= 1u << s;
            else if (lane == 0) x.failed = 1 + s;
            return here;
        };
        // the service warp's: the word's bits of token t, and the counters
        uint4 wb[kSplitMapWords / 128];
        auto load_bits = [&](int t) {
            const uint32_t *row = a.bits + static_cast<int64_t>(rec_of(t)[1].z) * a.KWp;
#pragma unroll
            for (int i = 0; i < kSplitMapWords / 128; ++i)
                wb[i] = 128 * i + 4 * lane < a.KWp ? *reinterpret_cast<const uint4 *>(row + 128 * i + 4 * lane) : make_uint4(0u, 0u, 0u, 0u);
        };
        int znew = 0;
        uint32_t c_min = 0, c_cnt = 0, c_int = 0;
        auto flip = [&](int p) {
            const int k = form.topic(p), w = k >> 5;
            if (((w >> 2) & 31) == lane) map[w] ^= 1u << (k & 31);
        };
        auto count = [&](int t) {
            const uint4 t1 = rec_of(t)[1];
            const int n_w = static_cast<int>(t1.w & 0xFFFFu), drawn = x.drawn[t & 1];
            const bool born = x.born[t & 3] != 0, died = x.died[t & 3] != 0;
            if (born) flip(prev);
            if (died) flip(static_cast<int>(t1.w >> 16));
            kd += (born ? 1 : 0) - (died ? 1 : 0);
            c_min += static_cast<uint32_t>(kd < n_w ? kd : n_w);
            c_cnt += (kd < n_w ? 1u : 0u) + (drawn & kDrawnAlias ? 1u << 6 : 0u) + (drawn & kDrawnZero ? 1u << 12 : 0u);
#pragma unroll
            for (int i = 0; i < kSplitMapWords / 128; ++i) {
                const uint4 mb = *reinterpret_cast<const uint4 *>(map + 128 * i + 4 * lane);
                c_int += static_cast<uint32_t>(__popc(wb[i].x & mb.x) + __popc(wb[i].y & mb.y) + __popc(wb[i].z & mb.z) + __popc(wb[i].w & mb.w));
            }
            prev = drawn & 0x3FFF;
            const int tt = t & 31;
            if (lane == tt) znew = prev;
            if (tt == 31 || t + 1 == n) {
                if (lane <= tt) r.z[p0 + t - tt + lane] = static_cast<int16_t>(guard_index(form.topic(znew), K, a.stats));
                add_block_counts(x.cnt, lane, tt + 1, c_min, c_cnt, c_int);
                c_min = c_cnt = c_int = 0;
            }
        };
        // the last warp's: token t's column, if it is short, padded to whole threads
        auto bring_column = [&](int t) {
            if (t >= n || *row_of(t) != 0xFFFFFFFFu) return;
            const uint4 t0 = rec_of(t)[0];
            const int n_w = static_cast<int>(rec_of(t)[1].w & 0xFFFFu);
            if (n_w > kSplitColumn) return;
            const int64_t col = static_cast<int64_t>((static_cast<u64>(t0.y & 0xFFFFu) << 32) | t0.x);
            uint32_t *q = reinterpret_cast<uint32_t *>(col_of(t));
            uint16_t *p = reinterpret_cast<uint16_t *>(q + kSplitColumn);
            for (int j0 = 0; j0 < n_w; j0 += 256) {
                uint32_t qv[8];
                int k[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int j = j0 + 32 * i + lane;
                    qv[i] = j < n_w ? a.q[col + j] : 0u;
                    k[i] = j < n_w ? a.topic[col + j] : 0;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int j = j0 + 32 * i + lane;
                    if (j < ((n_w + 3) & ~3)) {
                        q[j] = qv[i];
                        p[j] = static_cast<uint16_t>(pos(guard_index(k[i], K, a.stats)));
                    }
                }
            }
        };
        const int e = kSplitWarps * lane + warp;        // a thread's place in topic order
        // the last token's topic into the counts
        auto bring_in = [&](int t) {
            if (due >= 0 && mine(due)) {
                const uint32_t c = m.get(due) + 1u;
                m.set(due, c);
                if (c == 256u || c == 65536u) {
                    m.lvl = max(m.lvl, count_level(c));
                    atomicMax(&x.high, m.lvl);
                }
                x.born[t & 3] = c == 1;
            }
        };
        // the next token's record, and its own topic out of the counts
        uint4 n0, n1;
        uint32_t nd;
        auto read_record = [&](int t) {
            n0 = rec_of(t)[0];
            n1 = rec_of(t)[1];
            nd = *row_of(t);
        };
        auto take_out = [&](int t) {
            const int kold = static_cast<int>(n1.w >> 16);
            if (mine(kold)) {
                const uint32_t c = m.get(kold) - 1u;
                m.set(kold, c);
                x.died[t & 3] = c == 0;
            }
        };
        __syncthreads();            // the last pass's topics are written
        if (warp == kSplitWarps)
            for (int step = 0; step < 3; ++step) stage(0, step);
        __syncthreads();
        if (warp == kSplitWarps) {
            if (lane == 0) {
                fetch(0);
                fetch(1);
            }
            __syncwarp();
            if (!landed(0)) x.bad[0] = 1;
        }
        if (warp > kSplitWarps) bring_column(0);
        if (!service) {
            // before the first token's own topic goes out: that may be the same token again
            if (prev < 0 && threadIdx.x == 0) x.born[0] = 0;
            bring_in(0);
            due = -1;
            read_record(0);
            take_out(0);
        }
        __syncthreads();
        int done = 0, slot = 0;     // slot = t % 3
        for (int t = 0; t < n; ++t) {
            const int tt = t & 31;
            if (warp > kSplitWarps) {
                bring_column(t + 1);
            } else if (service) {
                if (lane == 0) fetch(t + 2);
                if (t > 0) count(t - 1);
                load_bits(t);
                if ((t | 31) + 1 < n && (tt & 7) == 0 && tt < 24) stage((t >> 5) + 1, tt >> 3);
                if (!landed(t + 1)) x.bad[t & 1] = 1;
                if (lane == 0 && (tt == 31 || t + 1 == n)) x.halt[t & 1] = r.deadline != ~0ull && global_ns() >= r.deadline ? 1 : 0;
            } else {
                const uint4 t0 = n0, t1 = n1;
                const uint32_t d = nd;
                if (t + 1 < n) read_record(t + 1);
                const int high = x.high;
                TokenDraw td;
                td.kold = static_cast<int>(t1.w >> 16);
                td.At = (static_cast<u64>(t0.w) << 32) | t0.z;
                td.U = (static_cast<u64>(t1.x) << 32) | t1.y;
                td.ka = static_cast<int>(t0.y >> 16);
                const int n_w = static_cast<int>(t1.w & 0xFFFFu);
                const bool dense = d != 0xFFFFFFFFu, brief = !dense && n_w <= kSplitColumn;
                const int seg = brief ? kSplitEntries : (n_w + 32 * kSplitWarps - 1) / (32 * kSplitWarps);
                const int j0 = min(seg * e, n_w), j1 = min(j0 + seg, n_w);
                const int64_t col = static_cast<int64_t>((static_cast<u64>(t0.y & 0xFFFFu) << 32) | t0.x);
                const uint8_t *row = ring + slot * RB;
                u64 acc = 0, term[kSplitEntries] = {};
                int at[kSplitEntries] = {};
                if (!brief) bring_in(t);
                if (dense) {
                    for (int pl = 0; pl <= m.lvl; ++pl) {
                        uint32_t s0 = 0, s1 = 0, s2 = 0;        // at most 128 topics of 255^2 each
                        const uint8_t *mp = counts + pl * PB + 16 * lane, *rp = row + 16 * lane;
#pragma unroll 4
                        for (int c = c0; c < c1; ++c) {
                            const uint4 w = *reinterpret_cast<const uint4 *>(mp + 512 * c);
                            const uint4 a0 = *reinterpret_cast<const uint4 *>(rp + 512 * c);
                            const uint4 a1 = *reinterpret_cast<const uint4 *>(rp + 512 * c + PB);
                            const uint4 a2 = *reinterpret_cast<const uint4 *>(rp + 512 * c + 2 * PB);
                            s0 = __dp4a(w.x, a0.x, s0); s1 = __dp4a(w.x, a1.x, s1); s2 = __dp4a(w.x, a2.x, s2);
                            s0 = __dp4a(w.y, a0.y, s0); s1 = __dp4a(w.y, a1.y, s1); s2 = __dp4a(w.y, a2.y, s2);
                            s0 = __dp4a(w.z, a0.z, s0); s1 = __dp4a(w.z, a1.z, s1); s2 = __dp4a(w.z, a2.z, s2);
                            s0 = __dp4a(w.w, a0.w, s0); s1 = __dp4a(w.w, a1.w, s1); s2 = __dp4a(w.w, a2.w, s2);
                        }
                        acc += (static_cast<u64>(s0) + (static_cast<u64>(s1) << 8) + (static_cast<u64>(s2) << 16)) << (8 * pl);
                    }
                } else if (brief) {
                    // the last token's topic is not in the counts yet: added where an entry names it
                    if (j0 < n_w) {
                        const uint4 q = *reinterpret_cast<const uint4 *>(col_of(t) + 16 * e);
                        const uint2 p = *reinterpret_cast<const uint2 *>(col_of(t) + 4 * kSplitColumn + 8 * e);
                        at[0] = static_cast<int>(p.x & 0xFFFFu);
                        at[1] = static_cast<int>(p.x >> 16);
                        at[2] = static_cast<int>(p.y & 0xFFFFu);
                        at[3] = static_cast<int>(p.y >> 16);
                        uint32_t c[kSplitEntries];
#pragma unroll
                        for (int i = 0; i < kSplitEntries; ++i) c[i] = counts[at[i]];
                        for (int pl = 1; pl <= high; ++pl)
#pragma unroll
                            for (int i = 0; i < kSplitEntries; ++i) c[i] |= static_cast<uint32_t>(counts[at[i] + pl * PB]) << (8 * pl);
#pragma unroll
                        for (int i = 0; i < kSplitEntries; ++i) c[i] += at[i] == due ? 1u : 0u;
                        term[0] = static_cast<u64>(q.x) * c[0];
                        term[1] = static_cast<u64>(q.y) * c[1];
                        term[2] = static_cast<u64>(q.z) * c[2];
                        term[3] = static_cast<u64>(q.w) * c[3];
                        acc = (term[0] + term[1]) + (term[2] + term[3]);
                    }
                } else {
                    split_barrier();        // every thread's counts are up to date
#pragma unroll 1
                    for (int j = j0; j < j1; ++j)
                        acc += static_cast<u64>(a.q[col + j]) * all.get(pos(guard_index(a.topic[col + j], K, a.stats)));
                }
                x.part[e] = acc;
                split_barrier();            // A
                const ulonglong2 s01 = *reinterpret_cast<const ulonglong2 *>(&x.part[kSplitWarps * lane]);
                const ulonglong2 s23 = *reinterpret_cast<const ulonglong2 *>(&x.part[kSplitWarps * lane + 2]);
                const u64 sum = s01.x + s01.y + s23.x + s23.y;
                const u64 incl = warp_incl_scan<32>(sum);
                const u64 T = td.At + (__shfl_sync(0xFFFFFFFFu, incl, 31) << kFracBits);
                const u64 rr = __umul64hi(td.U, T);
                const u64 rb = (rr - td.At) >> kFracBits;
                // no lane passes for an alias draw (rr < At wraps round) or without any mass
                const uint32_t bal = __ballot_sync(0xFFFFFFFFu, rb < incl);
                if (bal == 0) {
                    if (threadIdx.x == 0) x.drawn[t & 1] = static_cast<int>(rr < td.At ? td.ka | kDrawnAlias : td.kold | kDrawnZero);
                } else {
                    const int L = __ffs(bal) - 1;
                    u64 res = rb - (incl - sum);
                    int w = 0;
                    if (res >= s01.x) { res -= s01.x; w = 1; }
                    if (w == 1 && res >= s01.y) { res -= s01.y; w = 2; }
                    if (w == 2 && res >= s23.x) { res -= s23.x; w = 3; }
                    w = __shfl_sync(0xFFFFFFFFu, w, L);
                    if (w == warp) {
                        res = __shfl_sync(0xFFFFFFFFu, res, L);
                        int found = -1;
                        if (dense) {
                            // lane L's topics of this warp's chunks, four per lane
                            const int c = c0 + (lane >> 2), p = 512 * c + 16 * L + 4 * (lane & 3);
                            const int lvl = __shfl_sync(0xFFFFFFFFu, m.lvl, L);
                            uint32_t q[3] = {0u, 0u, 0u}, cw[3] = {0u, 0u, 0u};
                            if (c < c1) {
#pragma unroll
                                for (int i = 0; i < 3; ++i) {
                                    q[i] = *reinterpret_cast<const uint32_t *>(row + i * PB + p);
                                    if (i <= lvl) cw[i] = *reinterpret_cast<const uint32_t *>(counts + i * PB + p);
                                }
                            }
                            u64 t4[4], four = 0;
#pragma unroll
                            for (int b = 0; b < 4; ++b) {
                                const uint32_t qb = __byte_perm(__byte_perm(q[0], q[1], b | ((4 + b) << 4)), q[2], 0x0010 | ((4 + b) << 8)) & 0xFFFFFFu;
                                const uint32_t mc = __byte_perm(__byte_perm(cw[0], cw[1], b | ((4 + b) << 4)), cw[2], 0x0010 | ((4 + b) << 8)) & 0xFFFFFFu;
                                t4[b] = static_cast<u64>(qb) * mc;
                                four += t4[b];
                            }
                            const u64 in4 = warp_incl_scan<32>(four);
                            const uint32_t f = __ballot_sync(0xFFFFFFFFu, res < in4);
                            if (f && lane == __ffs(f) - 1) {
                                u64 run = in4 - four;
                                int b = 0;
#pragma unroll
                                for (int i = 0; i < 3; ++i) {
                                    run += t4[i];
                                    if (res >= run) b = i + 1;
                                }
                                x.drawn[t & 1] = p + b;
                            }
                            found = f ? 0 : -1;
                        } else if (lane == L) {
                            if (brief) {
#pragma unroll
                                for (int i = kSplitEntries - 1; i >= 0; --i) {
                                    u64 upto = 0;
#pragma unroll
                                    for (int j = 0; j <= i; ++j) upto += term[j];
                                    if (res < upto) found = at[i];
                                }
                            } else {
#pragma unroll 1
                                for (int j = j0; j < j1; ++j) {
                                    const int k = pos(guard_index(a.topic[col + j], K, a.stats));
                                    const u64 p = static_cast<u64>(a.q[col + j]) * all.get(k);
                                    if (res < p) { found = k; break; }
                                    res -= p;
                                }
                            }
                            if (found >= 0) x.drawn[t & 1] = found;
                        }
                        if (found < 0 && lane == L) {
                            atomicOr(&a.stats[ST_ERROR], ERR_INTERNAL);
                            x.drawn[t & 1] = td.kold;
                        }
                    }
                }
                if (brief) bring_in(t);
                else if (!dense) split_barrier();       // the counts of a long column are read
                if (t + 1 < n) take_out(t + 1);
            }
            __syncthreads();                // B
            ok = x.bad[t & 1] == 0;
            if (!ok) break;
            if (!service) due = prev = x.drawn[t & 1] & 0x3FFF;
            done = t + 1;
            slot = slot == 2 ? 0 : slot + 1;
            if ((tt == 31 || t + 1 == n) && x.halt[t & 1] != 0) {
                stop = true;
                break;
            }
        }
        if (warp == kSplitWarps && done > 0 && ok) count(done - 1);
        // the copy in flight where the pass ended early
        if (warp == kSplitWarps && !landed(done + (ok ? 1 : 2))) ok = false;
        if (!ok) stop = true;
        r.budget -= done;
        r.pos += done;
        if (r.pos == r.len) { r.pos = 0; r.sweep += 1; }
    }
    __syncthreads();
    if (warp == kSplitWarps && x.failed) cta_failed(a, x, phases);
}

}  // namespace pulda
