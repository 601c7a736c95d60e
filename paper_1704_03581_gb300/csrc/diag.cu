// The log-posterior diagnostic of the paper's experiments (Section 5, the
// log-posterior trace plots): the collapsed log joint of the topic indicators
// and the words, with Theta and Phi integrated out of the Dirichlet-
// multinomial LDA model,
//
//   log p(w, z | alpha, beta)
//     = sum_d [ lgamma(A) - lgamma(A + N_d) + sum_k ( lgamma(alpha_k + m_{d,k}) - lgamma(alpha_k) ) ]
//     + sum_k [ lgamma(V beta) - lgamma(V beta + n_k) + sum_v ( lgamma(beta + n_{k,v}) - lgamma(beta) ) ],
//
// A = sum_k alpha_k, n_k = sum_v n_{k,v}; terms with a zero count vanish.
// A table of the small-count terms, one warp per document (m_d in shared
// memory), one warp per word (the word's n column, rebuilt from z by the
// Phi-step's count pass), the rows' terms, and one CTA that adds the partial
// sums.  Every lane adds its own terms in a fixed order and so does each later
// step, so the same topics always give the same bits.  The GPU has few FP64
// units, and FP64 additions bound the passes: so no warp sum per document or
// word, and a document's terms are taken off a list of its topics, 32 at a
// time, not off all K (37,500 documents of 330 tokens, K = 1000: 227 -> 56 us;
// 100,000 words 133 -> 78 us; one CTA's final sums and lgammas 76 -> 20 us).
#include <algorithm>
#include <cstdint>

#include "pulda_internal.h"

namespace pulda {
namespace {

constexpr int kDiagWarps = 8;
// Most counts are small: the terms lgamma(alpha_k + c) - lgamma(alpha_k) for
// c < kTabA and lgamma(beta + n) - lgamma(beta) for n < kTabB are tabulated
// once per evaluation, with the same expression, so each term keeps its bits.
constexpr int kTabA = 256;
constexpr int kTabB = 4096;

// ta[k * kTabA + c] = lgamma(alpha_k + c) - lgamma(alpha_k);  tb[n] = lgamma(beta + n) - lgamma(beta).
// lgamma is FP64 work: a row per CTA shares lgamma(alpha_k), a symmetric
// alpha (rows = 1) has one row for every topic, and what every warp of the
// other passes needs is computed here once: lg = lgamma of beta, A, V beta.
__global__ void __launch_bounds__(kTabA) k_lp_tables(const float *alpha, int rows, double beta, double asum, double vb,
                                                     double *ta, double *tb, double *lg) {
    __shared__ double base;
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x < 3) lg[threadIdx.x] = lgamma(threadIdx.x == 0 ? beta : threadIdx.x == 1 ? asum : vb);
    for (int r = blockIdx.x; r < rows + kTabB / kTabA; r += gridDim.x) {
        const bool of_alpha = r < rows;
        const double x0 = of_alpha ? static_cast<double>(alpha[r]) : beta;
        const int n = of_alpha ? threadIdx.x : (r - rows) * kTabA + threadIdx.x;
        if (threadIdx.x == 0) base = lgamma(x0);
        const double top = lgamma(x0 + static_cast<double>(n));
        __syncthreads();
        (of_alpha ? ta + static_cast<int64_t>(r) * kTabA : tb)[n] = top - base;
        __syncthreads();
    }
}

// Butterfly sum: every lane ends with the same, order-fixed value.
__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// A warp's counts, the bitmap of its document's topics, and their list.
__host__ __device__ __forceinline__ int lp_doc_words(int K) { return K + (K + 31) / 32 + (K + 1) / 2; }

// doc_part[warp] = its documents' lgamma(A) - lgamma(A + N_d) +
// sum_{k: m_{d,k} > 0} (lgamma(alpha_k + m_{d,k}) - lgamma(alpha_k)).
// Documents are assigned to warps statically; the lgamma(A + N_d) of up to 32
// of them wait for one evaluation, a document per lane.
constexpr int kDocLoads = 8;
__global__ void k_lp_docs(const int64_t *doc_off, int64_t D, const int16_t *z, int K, const float *alpha, double asum,
                          const double *ta, const double *lg, int row, double *doc_part) {
    extern __shared__ uint32_t dsm[];
    const int lane = threadIdx.x & 31, KW = (K + 31) / 32;
    uint32_t *m = dsm + static_cast<size_t>(threadIdx.x >> 5) * lp_doc_words(K);
    uint32_t *bits = m + K;
    uint16_t *list = reinterpret_cast<uint16_t *>(bits + KW);
    const int warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
    for (int k = lane; k < K + KW; k += 32) m[k] = 0;
    __syncwarp();
    const double lga = lg[1];
    double acc = 0.0;
    int held = 0;
    int64_t held_n = 0;
    auto flush = [&] {
        if (lane < held) acc += lga - lgamma(asum + static_cast<double>(held_n));
        held = 0;
    };
    auto add = [&](int k) {
        if (atomicAdd(&m[k], 1u) == 0) atomicOr(&bits[k >> 5], 1u << (k & 31));
    };
    for (int64_t d = warp; d < D; d += warps) {
        const int64_t b = doc_off[d], e = doc_off[d + 1];
        int64_t i = b + lane;
        for (; i + 32 * (kDocLoads - 1) < e; i += 32 * kDocLoads) {
            int zz[kDocLoads];
#pragma unroll
            for (int u = 0; u < kDocLoads; ++u) zz[u] = z[i + 32 * u];
#pragma unroll
            for (int u = 0; u < kDocLoads; ++u) add(zz[u]);
        }
        for (; i < e; i += 32) add(z[i]);
        __syncwarp();
        int n = 0;                                     // the topics, ascending
        for (int w0 = 0; w0 < KW; w0 += 32) {
            const int w = w0 + lane;
            uint32_t x = w < KW ? bits[w] : 0u;
            if (w < KW) bits[w] = 0;
            int at = __popc(x);
            const int own = at;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xFFFFFFFFu, at, o);
                if (lane >= o) at += y;
            }
            uint16_t *l = list + n + at - own;
            for (; x; x &= x - 1u) *l++ = static_cast<uint16_t>(32 * w + __ffs(x) - 1);
            n += __shfl_sync(0xFFFFFFFFu, at, 31);
        }
        __syncwarp();
#pragma unroll 4
        for (int j = lane; j < n; j += 32) {
            const int k = list[j];
            const uint32_t c = m[k];
            m[k] = 0;
            if (c < kTabA) {
                acc += ta[static_cast<int64_t>(k) * row + c];
            } else {
                const double ak = static_cast<double>(alpha[k]);
                acc += lgamma(ak + static_cast<double>(c)) - lgamma(ak);
            }
        }
        if (lane == held) held_n = e - b;
        if (++held == 32) flush();
        __syncwarp();
    }
    flush();
    acc = warp_sum_f64(acc);
    if (lane == 0) doc_part[warp] = acc;
}

// word_part[warp] = its words' sum_{k: n_{k,v} > 0} (lgamma(beta + n_{k,v}) - lgamma(beta));
// n_k accumulated (integer atomics, so in any order; a CTA's in shared memory
// first where K counts fit).  Words are assigned to warps statically, but the
// n_heavy most frequent ones (heavy_row >= 0), whose counts are past the table
// and whose columns are long, in pieces of 32 entries.
__global__ void k_lp_words(const int32_t *word_order, const int32_t *heavy_row, int n_heavy, int K, const int64_t *word_off, const uint16_t *nst_k, const uint32_t *nst_n,
                           const int32_t *nnz_n, int V, double beta, const double *tb, const double *lg, double *word_part,
                           unsigned long long *nk, int k_shared) {
    extern __shared__ uint32_t nsm[];
    const int lane = threadIdx.x & 31;
    const int warps = gridDim.x * (blockDim.x >> 5), warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const double lgb = lg[0];
    for (int k = threadIdx.x; k < k_shared; k += blockDim.x) nsm[k] = 0;
    __syncthreads();
    double acc = 0.0;
    auto entry = [&](int64_t at) {
        const uint32_t n = nst_n[at];
        const int k = nst_k[at];
        acc += n < static_cast<uint32_t>(kTabB) ? tb[n] : lgamma(beta + static_cast<double>(n)) - lgb;
        if (k_shared) atomicAdd(&nsm[k], n);               // fewer than 2^31 tokens
        else atomicAdd(&nk[k], static_cast<unsigned long long>(n));
    };
    const int pieces = (K + 31) / 32;
    for (int64_t i = warp; i < static_cast<int64_t>(n_heavy) * pieces; i += warps) {
        const int v = word_order[i / pieces], j = 32 * static_cast<int>(i % pieces) + lane;
        if (j < nnz_n[v]) entry(word_off[v] + j);
    }
    for (int v = warp; v < V; v += warps) {
        if (n_heavy > 0 && heavy_row[v] >= 0) continue;
        const int64_t b = word_off[v];
        const int cnt = nnz_n[v];
#pragma unroll 4
        for (int j = lane; j < cnt; j += 32) entry(b + j);
    }
    acc = warp_sum_f64(acc);
    if (lane == 0) word_part[warp] = acc;
    __syncthreads();
    for (int k = threadIdx.x; k < k_shared; k += blockDim.x)
        if (nsm[k]) atomicAdd(&nk[k], static_cast<unsigned long long>(nsm[k]));
}

// row_lp[k] = lgamma(V beta) - lgamma(V beta + n_k).
__global__ void __launch_bounds__(32) k_lp_rows(const unsigned long long *nk, int K, double vb, const double *lg, double *row_lp) {
    const int k = blockIdx.x * 32 + threadIdx.x;
    if (k < K) row_lp[k] = lg[2] - lgamma(vb + static_cast<double>(nk[k]));
}

// A sum with the rounding errors of its additions kept beside it (Knuth's
// two-sum): the last, largest additions would otherwise decide the error.
struct Sum2 {
    double s, e;
    __device__ __forceinline__ void add(double x) {
        const double t = s + x, y = t - s;
        e += (s - (t - y)) + (x - y);
        s = t;
    }
    __device__ __forceinline__ void add(const Sum2 &o) {
        add(o.s);
        e += o.e;
    }
    __device__ __forceinline__ double value() const { return s + e; }
};

// out = {total, document sum, topic sum}: each thread adds a fixed strided
// slice in order, then a fixed tree.
constexpr int kFinalThreads = 512;
__global__ void __launch_bounds__(kFinalThreads) k_lp_final(const double *doc_part, int nd, const double *word_part,
                                                            int nw, const double *row_lp, int K, double *out) {
    __shared__ Sum2 sd[kFinalThreads], st[kFinalThreads];
    const int t = threadIdx.x;
    Sum2 a{0.0, 0.0}, b{0.0, 0.0};
#pragma unroll 8
    for (int i = t; i < nd; i += kFinalThreads) a.add(doc_part[i]);
#pragma unroll 8
    for (int i = t; i < nw; i += kFinalThreads) b.add(word_part[i]);
    for (int k = t; k < K; k += kFinalThreads) b.add(row_lp[k]);
    sd[t] = a;
    st[t] = b;
    __syncthreads();
    for (int s = kFinalThreads / 2; s > 0; s >>= 1) {
        if (t < s) {
            sd[t].add(sd[t + s]);
            st[t].add(st[t + s]);
        }
        __syncthreads();
    }
    if (t == 0) {
        out[1] = sd[0].value();
        out[2] = st[0].value();
        sd[0].add(st[0]);
        out[0] = sd[0].value();
    }
}

int device_attr(cudaDeviceAttr what) {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, what, dev);
    return v;
}

}  // namespace

size_t log_posterior_scratch_bytes(int64_t D, int V, int K) {
    // the warps of the document pass are at most D + kDiagWarps, those of the word pass V + 32
    return sizeof(double) * (static_cast<size_t>(D) + kDiagWarps + static_cast<size_t>(V) + 32 + 6 + static_cast<size_t>(K) * (kTabA + 1) + kTabB) +
           sizeof(unsigned long long) * static_cast<size_t>(K);
}

void launch_log_posterior(const int64_t *doc_off, int64_t D, const int16_t *z, int K, const float *alpha, double asum,
                          const PhiArgs &counts, double beta, bool symmetric, void *scratch, cudaStream_t st) {
    double *out = static_cast<double *>(scratch);
    double *lg = out + 3;
    double *doc_part = lg + 3;
    double *word_part = doc_part + D + kDiagWarps;
    double *row_lp = word_part + counts.V + 32;
    double *ta = row_lp + K;
    double *tb = ta + static_cast<size_t>(K) * kTabA;
    unsigned long long *nk = reinterpret_cast<unsigned long long *>(tb + kTabB);
    cudaMemsetAsync(nk, 0, sizeof(unsigned long long) * static_cast<size_t>(K), st);
    const int sms = std::max(1, device_attr(cudaDevAttrMultiProcessorCount));
    const int rows = symmetric ? 1 : K;
    k_lp_tables<<<std::min(rows + kTabB / kTabA, 8 * sms), kTabA, 0, st>>>(alpha, rows, beta, asum, static_cast<double>(counts.V) * beta, ta, tb, lg);
    int doc_warps = 0;
    if (D > 0) {
        // the CTA shrinks for large K
        int warps = kDiagWarps;
        const int optin = std::max(48 * 1024, device_attr(cudaDevAttrMaxSharedMemoryPerBlockOptin));
        while (warps > 1 && static_cast<size_t>(warps) * lp_doc_words(K) * sizeof(uint32_t) > static_cast<size_t>(optin)) warps >>= 1;
        const size_t smem = static_cast<size_t>(warps) * lp_doc_words(K) * sizeof(uint32_t);
        if (smem > 48 * 1024) cudaFuncSetAttribute(k_lp_docs, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lp_docs, 32 * warps, smem);
        const int64_t need = (D + warps - 1) / warps;
        const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(need, static_cast<int64_t>(sms) * std::max(1, per_sm))));
        k_lp_docs<<<grid, 32 * warps, smem, st>>>(doc_off, D, z, K, alpha, asum, ta, lg, symmetric ? 0 : kTabA, doc_part);
        doc_warps = grid * warps;
    }
    constexpr int kWordThreads = 1024;
    const int64_t words_cta = kWordThreads / 32;
    const int wgrid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((counts.V + words_cta - 1) / words_cta, 2LL * sms)));
    const int k_shared = K <= 12288 ? K : 0;               // within 48 KB
    k_lp_words<<<wgrid, kWordThreads, sizeof(uint32_t) * k_shared, st>>>(counts.word_order, counts.heavy_row, counts.n_heavy, K, counts.word_off, counts.nst_k, counts.nst_n, counts.nnz_n,
                                                                         counts.V, beta, tb, lg, word_part, nk, k_shared);
    k_lp_rows<<<(K + 31) / 32, 32, 0, st>>>(nk, K, static_cast<double>(counts.V) * beta, lg, row_lp);
    k_lp_final<<<1, kFinalThreads, 0, st>>>(doc_part, doc_warps, word_part, wgrid * static_cast<int>(words_cta), row_lp, K, out);
}

}  // namespace pulda
