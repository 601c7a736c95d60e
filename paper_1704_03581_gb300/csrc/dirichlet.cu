// Dirichlet Phi-step of the partially collapsed sampler (Algorithm 1), the
// method the Polya urn approximates: phi_k ~ Dir(n_k + beta) through the
// Gamma representation gamma_{k,v} ~ G(beta + n_{k,v}, 1), phi_{k,v} =
// gamma_{k,v} / sum_v gamma_{k,v} ("Efficient sampling of Phi": Gammas by
// Marsaglia and Tsang, 2000).  Every entry of the K x V matrix is drawn --
// the dense work the Polya urn's skip-ahead avoids.
//
// Readings, shared with the CPU oracle and implemented here independently:
//   Gamma draws in float, each operation rounded to float (explicit _rn
//   intrinsics); normals from the rounded-normal table; uniforms with 23
//   bits, u = (2 floor(x / 2^9) + 1) 2^-24; Philox counter (v, k, sweep,
//   TAG_GAMMA << 28 | attempt) per attempt and (v, k, sweep, TAG_GAMMA_BOOST
//   << 28) for the boost u^(1/a) of shapes a < 1; log and exp are this
//   file's own.  S_k is summed in double over chunks of kDirChunk words in
//   ascending order (each chunk in ascending v).  phi = gamma (1 / S_k) in
//   double; an entry stays in its column iff its 24-bit fixed-point weight
//   relative to the column maximum rounds to at least 1.
#include <algorithm>
#include <cstdint>

#include "device_rng.cuh"
#include "pulda_internal.h"

namespace pulda {
namespace {

using u64 = unsigned long long;

// ln x for finite x > 0: x = m 2^e with m in [sqrt(1/2), sqrt(2)], ln m =
// 2 atanh(s) with s = (m - 1) / (m + 1) (|s| <= 0.1716) by its series to s^9,
// ln 2 split in a short high part and a correction.
__device__ float own_logf(float x) {
    int e = 0;
    uint32_t b = __float_as_uint(x);
    if (b < 0x00800000u) {               // subnormal: scale by 2^24
        x = __fmul_rn(x, 16777216.0f);
        b = __float_as_uint(x);
        e = -24;
    }
    e += static_cast<int>(b >> 23) - 127;
    float m = __uint_as_float((b & 0x007FFFFFu) | 0x3F800000u);
    if (m > 1.41421354f) {
        m = __fmul_rn(m, 0.5f);
        e += 1;
    }
    const float s = __fdiv_rn(__fsub_rn(m, 1.0f), __fadd_rn(m, 1.0f));
    const float s2 = __fmul_rn(s, s);
    float t = __fmul_rn(s2, 0.222222224f);          // 2/9
    t = __fmul_rn(s2, __fadd_rn(0.285714298f, t));  // 2/7
    t = __fmul_rn(s2, __fadd_rn(0.400000006f, t));  // 2/5
    t = __fmul_rn(s2, __fadd_rn(0.666666687f, t));  // 2/3
    const float poly = __fmul_rn(s, __fadd_rn(2.0f, t));
    const float ef = static_cast<float>(e);
    return __fadd_rn(__fmul_rn(ef, 0.693359375f), __fadd_rn(__fmul_rn(ef, -2.12194442e-4f), poly));
}

// e^x for x <= 88: x = k ln 2 + r with |r| <= ln 2 / 2, e^r by its Taylor
// series to r^7, times 2^k (in two steps below 2^-126); 0 below -104.
__device__ float own_expf(float x) {
    if (x < -104.0f) return 0.0f;
    const float kf = floorf(__fadd_rn(__fmul_rn(x, 1.44269502f), 0.5f));
    const int k = static_cast<int>(kf);
    const float r = __fsub_rn(__fsub_rn(x, __fmul_rn(kf, 0.693359375f)), __fmul_rn(kf, -2.12194442e-4f));
    float p = __fmul_rn(r, 0.000198412701f);       // 1/5040
    p = __fmul_rn(r, __fadd_rn(0.00138888892f, p)); // 1/720
    p = __fmul_rn(r, __fadd_rn(0.00833333377f, p)); // 1/120
    p = __fmul_rn(r, __fadd_rn(0.0416666679f, p));  // 1/24
    p = __fmul_rn(r, __fadd_rn(0.166666672f, p));   // 1/6
    p = __fmul_rn(r, __fadd_rn(0.5f, p));
    p = __fmul_rn(r, __fadd_rn(1.0f, p));
    p = __fadd_rn(1.0f, p);
    if (k >= -126) return __fmul_rn(p, __uint_as_float(static_cast<uint32_t>(k + 127) << 23));
    return __fmul_rn(__fmul_rn(p, __uint_as_float(static_cast<uint32_t>(k + 64 + 127) << 23)),
                     __uint_as_float(static_cast<uint32_t>(127 - 64) << 23));
}

__device__ __forceinline__ float unif23(uint32_t x) {
    return __fmul_rn(static_cast<float>(2u * (x >> 9) + 1u), 5.96046448e-08f);   // 2^-24
}

// gauss_draw rounded to float.  Its five FP64 instructions were 81% of the
// FP64 pipe's time in the Gamma pass (0.75 ms for 50 M draws), so the
// interpolation runs in integers of 2^-58, whose value is within 2^-50 of the
// double's; where that does not settle the rounding to float (or next to 0)
// the double is computed.
__device__ __noinline__ float gauss_exact(const DevTables &T, uint32_t x0, uint32_t x1) { return __double2float_rn(gauss_draw(T, x0, x1)); }

__device__ __forceinline__ float gauss_float(const DevTables &T, uint32_t x0, uint32_t x1) {
    const uint32_t cell = x0 >> 16;
    const longlong2 node = T.gauss_fix[cell];                         // the cell's lower node and its width
    const long long a = node.x;
    const u64 step = static_cast<u64>(node.y);
    const long long x = a + static_cast<long long>(__umul64hi(step, (static_cast<u64>(x0 & 0xFFFFu) << 48) | (static_cast<u64>(x1) << 16)));
    const u64 mag = x < 0 ? 0ull - static_cast<u64>(x) : static_cast<u64>(x);
    const int sh = 40 - __clzll(static_cast<long long>(mag));         // bits below the 24 of a float
    if (sh >= 17) {
        const u64 half = 1ull << (sh - 1), rem = mag & (2 * half - 1);
        if (rem - half + 512 >= 1024) {
            const uint32_t q = static_cast<uint32_t>(mag >> sh) + (rem >= half ? 1u : 0u);
            const float r = __fmul_rn(static_cast<float>(q), __uint_as_float(static_cast<uint32_t>(sh - 58 + 127) << 23));
            return x < 0 ? -r : r;
        }
    }
    return gauss_exact(T, x0, x1);
}

// gamma ~ G(a, 1), a > 0, Marsaglia and Tsang; for a < 1 the draw of
// G(a + 1) is scaled by u^(1/a).
struct GammaShape { float a, d, cc; };
__device__ __forceinline__ GammaShape gamma_shape(float a) {
    const float sh = a < 1.0f ? __fadd_rn(a, 1.0f) : a;
    const float d = __fsub_rn(sh, 0.333333343f);
    return {a, d, __fdiv_rn(1.0f, __fsqrt_rn(__fmul_rn(9.0f, d)))};
}

// Attempt t: whether it is accepted (SQUEEZE: by the squeeze test alone), and its draw.
template <bool SQUEEZE>
__device__ __forceinline__ bool gamma_try(const DevTables &T, const GammaShape &s, uint64_t seed, uint32_t v, uint32_t k,
                                          uint32_t sweep, uint32_t t, float *r) {
    const U4 x = draw(seed, v, k, sweep, TAG_GAMMA, t);
    const float g = gauss_float(T, x.x, x.y);
    const float y = __fadd_rn(1.0f, __fmul_rn(s.cc, g));
    const float v3 = __fmul_rn(__fmul_rn(y, y), y);
    *r = __fmul_rn(s.d, v3);
    if (y <= 0.0f) return false;
    const float u = unif23(x.z);
    const float g2 = __fmul_rn(g, g);
    if (u < __fsub_rn(1.0f, __fmul_rn(0.0331f, __fmul_rn(g2, g2)))) return true;
    if (SQUEEZE) return false;
    return own_logf(u) < __fadd_rn(__fmul_rn(0.5f, g2), __fmul_rn(s.d, __fadd_rn(__fsub_rn(1.0f, v3), own_logf(v3))));
}

__device__ __forceinline__ float gamma_boost(const GammaShape &s, float r, uint64_t seed, uint32_t v, uint32_t k, uint32_t sweep) {
    if (!(s.a < 1.0f)) return r;
    const U4 xb = draw(seed, v, k, sweep, TAG_GAMMA_BOOST, 0);
    return __fmul_rn(r, own_expf(__fdiv_rn(own_logf(unif23(xb.x)), s.a)));
}

// *fail is set if no attempt was accepted.
__device__ float gamma_draw(const DevTables &T, const GammaShape &s, uint64_t seed, uint32_t v, uint32_t k, uint32_t sweep, bool *fail) {
    float r;
    for (uint32_t t = 0; t < kMaxGammaTry; ++t)
        if (gamma_try<false>(T, s, seed, v, k, sweep, t, &r)) return gamma_boost(s, r, seed, v, k, sweep);
    *fail = true;
    return 0.0f;
}

constexpr int kSelBlock = 128;

// A warp's counts of one word, and the list of its topics.
__host__ __device__ __forceinline__ int dir_gamma_words(int K) { return K + (K + 1) / 2; }

// One warp per word (grid-stride): the word's n column into a dense array in
// the warp's shared memory, then gamma_{k,v} for every topic, word-major.
// Warps do not wait on one another between words.  The pass is bound by
// instruction issue (every entry has one or two Philox blocks, a logarithm and
// an exponential), so the lanes first take the draws of the entries with n = 0
// that the squeeze test accepts at once, about nine in ten of a rare word's;
// the others, for which a whole warp would compute a shape's constants or run
// the logarithms and further attempts, are listed and drawn 32 at a time.
// 50 M draws: 1.13 ms before, 0.71 now; 2, 4 or 5 CTAs per SM instead of 3 cost
// 0.03 to 0.09 ms.
__global__ void __launch_bounds__(256, 3) k_dir_gamma(PhiArgs a) {
    extern __shared__ uint32_t nsm[];
    const int K = a.K;
    const int lane = threadIdx.x & 31;
    uint32_t *nrow = nsm + static_cast<size_t>(threadIdx.x >> 5) * dir_gamma_words(K);
    uint16_t *slow = reinterpret_cast<uint16_t *>(nrow + K);
    const int wpb = blockDim.x >> 5;
    const int nwarps = gridDim.x * wpb;
    const uint32_t sweep = a.sweep_ptr ? *a.sweep_ptr : a.sweep;
    const float bf = static_cast<float>(a.tab.beta);
    const GammaShape zero = gamma_shape(bf);
    bool fail = false;
    for (int v = blockIdx.x * wpb + (threadIdx.x >> 5); v < a.V; v += nwarps) {
        for (int k = lane; k < K; k += 32) nrow[k] = 0;
        __syncwarp();
        const int64_t b = a.word_off[v];
        for (int j = lane; j < a.nnz_n[v]; j += 32) nrow[a.nst_k[b + j]] = a.nst_n[b + j];
        __syncwarp();
        float *out = a.gam + static_cast<int64_t>(v) * K;
        int n_slow = 0;
        for (int k0 = 0; k0 < K; k0 += 32) {
            const int k = k0 + lane;
            bool ok = false;
            if (k < K && nrow[k] == 0) {
                float r;
                ok = gamma_try<true>(a.tab, zero, a.seed, static_cast<uint32_t>(v), static_cast<uint32_t>(k), sweep, 0, &r);
                r = gamma_boost(zero, r, a.seed, static_cast<uint32_t>(v), static_cast<uint32_t>(k), sweep);
                if (ok) out[k] = r;
            }
            const uint32_t bal = __ballot_sync(0xFFFFFFFFu, k < K && !ok);
            if (k < K && !ok) slow[n_slow + __popc(bal & ((1u << lane) - 1u))] = static_cast<uint16_t>(k);
            n_slow += __popc(bal);
        }
        __syncwarp();
        for (int i = lane; i < n_slow; i += 32) {
            const int k = slow[i];
            const GammaShape g = gamma_shape(__fadd_rn(bf, static_cast<float>(nrow[k])));
            out[k] = gamma_draw(a.tab, g, a.seed, static_cast<uint32_t>(v), static_cast<uint32_t>(k), sweep, &fail);
        }
        __syncwarp();
    }
    if (fail) atomicOr(&a.stats[ST_ERROR], ERR_GAMMA);
}

// dpart[c * K + k] = sum over the words of chunk c, in ascending order, of
// gamma_{k,v}: one thread per chunk and topic, whose loads (not its additions)
// go 16 at a time.
// FP64 bounds the pass, so a normal float is widened with integers (its bits,
// the exponent rebiased) and only the additions are FP64: 79% of that pipe's
// time, 0.21 ms for 50 M draws (0.29 before).
constexpr int kRowBlock = 128;
__device__ __forceinline__ double widen(float x) {            // x >= 0
    const uint32_t b = __float_as_uint(x);
    if (b < 0x00800000u || b >= 0x7F800000u) return static_cast<double>(x);
    return __hiloint2double(static_cast<int>((b >> 3) + (896u << 20)), static_cast<int>(b << 29));
}

__global__ void __launch_bounds__(kRowBlock) k_dir_rowsum_part(PhiArgs a) {
    const int K = a.K;
    const int c = blockIdx.x, k = blockIdx.y * kRowBlock + threadIdx.x;
    if (k >= K) return;
    const int v0 = c * kDirChunk, v1 = min(a.V, v0 + kDirChunk);
    double part = 0.0;
    int v = v0;
    for (; v + 15 < v1; v += 16) {
        float g[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) g[u] = a.gam[static_cast<int64_t>(v + u) * K + k];
#pragma unroll
        for (int u = 0; u < 16; ++u) part = __dadd_rn(part, widen(g[u]));
    }
    for (; v < v1; ++v) part = __dadd_rn(part, widen(a.gam[static_cast<int64_t>(v) * K + k]));
    a.dpart[static_cast<int64_t>(c) * K + k] = part;
}

// S_k = the chunk sums in ascending chunk order; 1 / S_k (0 for a row of zeros).
__global__ void __launch_bounds__(32) k_dir_rowsum_final(PhiArgs a, int n_chunks) {
    const int k = blockIdx.x * 32 + threadIdx.x;
    if (k >= a.K) return;
    double tot = 0.0;
    int c = 0;
    for (; c + 15 < n_chunks; c += 16) {
        double p[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) p[u] = a.dpart[static_cast<int64_t>(c + u) * a.K + k];
#pragma unroll
        for (int u = 0; u < 16; ++u) tot = __dadd_rn(tot, p[u]);
    }
    for (; c < n_chunks; ++c) tot = __dadd_rn(tot, a.dpart[static_cast<int64_t>(c) * a.K + k]);
    a.Sd[k] = tot;
    a.invS[k] = tot > 0.0 ? __ddiv_rn(1.0, tot) : 0.0;
    a.invSf[k] = __double2float_rn(a.invS[k]);
}

// One warp per word: phi = gamma (1/S_k) in double; the column maximum fixes
// the fixed-point scale 2^(24 - e); entries whose weight rounds to 0 are
// dropped, the rest staged in ascending topic order (cst_k, cst_c = the
// draw's bits).  FP64 is scarce on this GPU, so a float product screens every
// entry (relative error below 2^-22): the maximum is taken exactly over the
// entries within 2^-12 of the float maximum, and an entry is decided by the
// double test only within 0.1% of the threshold 2^(e-25).  Tiny columns (float
// maximum or threshold below 2^-100, where float products lose precision) take
// the double path throughout.  The decisions are those of the double test.
__global__ void k_dir_select(PhiArgs a) {
    const int lane = threadIdx.x & 31;
    const int K = a.K;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const float kTiny = 7.88860905e-31f;      // 2^-100
    for (int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < a.V; v += nwarps) {
        const float *g = a.gam + static_cast<int64_t>(v) * K;
        float fmax = 0.0f;
        for (int k = lane; k < K; k += 32) fmax = fmaxf(fmax, __fmul_rn(g[k], a.invSf[k]));
#pragma unroll
        for (int o = 16; o; o >>= 1) fmax = fmaxf(fmax, __shfl_xor_sync(0xFFFFFFFFu, fmax, o));
        const bool exact_all = fmax < kTiny;
        const float fcut = __fmul_rn(fmax, 0.999755859f);       // 1 - 2^-12
        double pmax = 0.0;
        for (int k = lane; k < K; k += 32) {
            if (exact_all || __fmul_rn(g[k], a.invSf[k]) >= fcut) {
                const double p = __dmul_rn(static_cast<double>(g[k]), a.invS[k]);
                pmax = p > pmax ? p : pmax;
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const double y = __shfl_xor_sync(0xFFFFFFFFu, pmax, o);
            pmax = y > pmax ? y : pmax;
        }
        int kept = 0;
        if (pmax > 0.0) {
            const long long bits = __double_as_longlong(pmax);
            const int e = static_cast<int>((bits >> 52) & 0x7FF) - 1022;
            const double scale = __longlong_as_double(static_cast<long long>(1023 + 24 - e) << 52);
            // threshold 2^(e-25) in float, when it is a normal float well above the subnormals
            const bool screen = !exact_all && e - 25 >= -100;
            const float thr = screen ? __uint_as_float(static_cast<uint32_t>(e - 25 + 127) << 23) : 0.0f;
            const float hi = __fmul_rn(thr, 1.001f), lo = __fmul_rn(thr, 0.999f);
            const int64_t dst = static_cast<int64_t>(v) * K;
            for (int k0 = 0; k0 < K; k0 += 32) {
                const int k = k0 + lane;
                bool keep = false;
                float gk = 0.0f;
                if (k < K) {
                    gk = g[k];
                    const float pf = screen ? __fmul_rn(gk, a.invSf[k]) : 0.0f;
                    if (screen && pf >= hi) {
                        keep = true;
                    } else if (!screen || pf > lo) {
                        const double p = __dmul_rn(static_cast<double>(gk), a.invS[k]);
                        keep = floor(__dadd_rn(__dmul_rn(p, scale), 0.5)) >= 1.0;
                    }
                }
                const uint32_t bal = __ballot_sync(0xFFFFFFFFu, keep);
                if (keep) {
                    const int at = kept + __popc(bal & ((1u << lane) - 1u));
                    a.cst_k[dst + at] = static_cast<uint16_t>(k);
                    a.cst_c[dst + at] = __float_as_uint(gk);
                }
                kept += __popc(bal);
            }
        }
        if (lane == 0) a.nnz_c[v] = kept;
    }
}

// The same up to 32 R topics (1,024 at most): the word's draws and products in
// registers, loaded at once, an entry's decisions as a bit each, and the few
// double products in loops of their own over those bits (short branches
// around them end up as FP64 instructions issued for every entry: 0.44 ms for
// 50,000 words of 1,000 topics; 0.19 with three passes over memory, 0.13 so).
template <int R>
__global__ void __launch_bounds__(kSelBlock, 5) k_dir_select_reg(PhiArgs a) {
    const int lane = threadIdx.x & 31;
    const int K = a.K;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const float kTiny = 7.88860905e-31f;      // 2^-100
    const uint32_t own = lane >= K ? 0u : 0xFFFFFFFFu >> (31 - (K - 1 - lane) / 32);     // bit i: topic 32 i + lane < K
    for (int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < a.V; v += nwarps) {
        const float *g = a.gam + static_cast<int64_t>(v) * K;
        float gr[R], pr[R];                   // 0 past K
#pragma unroll
        for (int i = 0; i < R; ++i) gr[i] = own >> i & 1u ? g[32 * i + lane] : 0.0f;
#pragma unroll
        for (int i = 0; i < R; ++i) pr[i] = own >> i & 1u ? __fmul_rn(gr[i], a.invSf[32 * i + lane]) : 0.0f;
        float fmax = 0.0f;
#pragma unroll
        for (int i = 0; i < R; ++i) fmax = fmaxf(fmax, pr[i]);
#pragma unroll
        for (int o = 16; o; o >>= 1) fmax = fmaxf(fmax, __shfl_xor_sync(0xFFFFFFFFu, fmax, o));
        const bool exact_all = fmax < kTiny;
        const float fcut = __fmul_rn(fmax, 0.999755859f);       // 1 - 2^-12
        uint32_t near = 0;
#pragma unroll
        for (int i = 0; i < R; ++i) near |= (pr[i] >= fcut ? 1u : 0u) << i;
        near = (exact_all ? 0xFFFFFFFFu : near) & own;
        double pmax = 0.0;
        for (; near; near &= near - 1u) {
            const int k = 32 * (__ffs(near) - 1) + lane;
            const double p = __dmul_rn(static_cast<double>(g[k]), a.invS[k]);
            pmax = p > pmax ? p : pmax;
        }
        // doubles >= 0 are ordered as their bits
        long long top = __double_as_longlong(pmax);
#pragma unroll
        for (int o = 16; o; o >>= 1) top = max(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
        int kept = 0;
        if (top > 0) {
            const int e = static_cast<int>(top >> 52) - 1022;
            const double scale = __longlong_as_double(static_cast<long long>(1023 + 24 - e) << 52);
            const bool screen = !exact_all && e - 25 >= -100;
            const float thr = screen ? __uint_as_float(static_cast<uint32_t>(e - 25 + 127) << 23) : 0.0f;
            const float hi = __fmul_rn(thr, 1.001f), lo = __fmul_rn(thr, 0.999f);
            uint32_t keep = 0, above = 0;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                keep |= (pr[i] >= hi ? 1u : 0u) << i;
                above |= (pr[i] > lo ? 1u : 0u) << i;
            }
            uint32_t test = screen ? above & ~keep : own;
            keep = screen ? keep & own : 0u;
            for (; test; test &= test - 1u) {
                const int i = __ffs(test) - 1, k = 32 * i + lane;
                const double p = __dmul_rn(static_cast<double>(g[k]), a.invS[k]);
                if (floor(__dadd_rn(__dmul_rn(p, scale), 0.5)) >= 1.0) keep |= 1u << i;
            }
            __syncwarp();
            const int64_t dst = static_cast<int64_t>(v) * K;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const bool mine = keep >> i & 1u;
                const uint32_t bal = __ballot_sync(0xFFFFFFFFu, mine);
                if (mine) {
                    const int at = kept + __popc(bal & ((1u << lane) - 1u));
                    a.cst_k[dst + at] = static_cast<uint16_t>(32 * i + lane);
                    a.cst_c[dst + at] = __float_as_uint(gr[i]);
                }
                kept += __popc(bal);
            }
        }
        if (lane == 0) a.nnz_c[v] = kept;
    }
}

int sms() {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

}  // namespace

size_t dir_part_count(int V, int K) {
    return static_cast<size_t>((V + kDirChunk - 1) / kDirChunk) * static_cast<size_t>(K);
}

void launch_dir_phi(const PhiArgs &a, cudaStream_t st) {
    const int n = sms();
    // one warp per word, its n row and topic list in shared memory: up to 8
    // warps per CTA within 96 KB (one warp of up to 96 KB for the largest K)
    int wpb = 8;
    while (wpb > 1 && static_cast<size_t>(wpb) * dir_gamma_words(a.K) * sizeof(uint32_t) > 96 * 1024) wpb >>= 1;
    const size_t smem = static_cast<size_t>(wpb) * dir_gamma_words(a.K) * sizeof(uint32_t);
    if (smem > 48 * 1024) {
        int dev = 0, optin = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        cudaFuncSetAttribute(k_dir_gamma, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    }
    const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((a.V + wpb - 1) / wpb, 16LL * n)));
    k_dir_gamma<<<grid, 32 * wpb, smem, st>>>(a);
    const int n_chunks = (a.V + kDirChunk - 1) / kDirChunk;
    k_dir_rowsum_part<<<dim3(n_chunks, (a.K + kRowBlock - 1) / kRowBlock), kRowBlock, 0, st>>>(a);
    k_dir_rowsum_final<<<(a.K + 31) / 32, 32, 0, st>>>(a, n_chunks);
    constexpr int W = kSelBlock / 32;
    const int sel_grid = std::max(1, std::min((a.V + W - 1) / W, 16 * n));
    auto select = a.K <= 256 ? k_dir_select_reg<8> : a.K <= 512 ? k_dir_select_reg<16> : a.K <= 1024 ? k_dir_select_reg<32> : k_dir_select;
    select<<<sel_grid, kSelBlock, 0, st>>>(a);
}

}  // namespace pulda
