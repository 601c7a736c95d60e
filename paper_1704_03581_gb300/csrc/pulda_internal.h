// Internal declarations of the pulda CUDA library (not part of the C ABI).
#pragma once
#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

namespace pulda {

// Alias tables are built for Poisson rates beta + l with l <= kL; larger
// counts use a rounded Gaussian ("Efficient sampling of Phi", L = 100).
constexpr int kL = 100;
// Length of the geometric-gap CDF table used to skip over entries whose
// Poisson rate is beta alone.
constexpr int kGeoLen = 1024;
// Equiprobable cells of the inverse-normal table.
constexpr int kGaussCells = 65536;
// The alpha part of the z conditional is held in units of 2^-16 q.
constexpr int kFracBits = 16;
// Dead-row redraw attempts before giving up.
constexpr uint32_t kMaxRedraw = 1u << 20;
// Largest K the kernels' shared-memory layouts accept.
constexpr int kMaxK = 16384;
// Bitmap rows are laid out for the grouped z-step's lanes up to here.
constexpr int kMaxKBitmap = 2048;
// Four documents per warp: each of a document's 8 lanes holds up to four
// words.
constexpr int kMaxKGrouped = 1024;
// Words of a word's bitmap row: ceil(K / 32) rounded up to 8 times a power
// of two, so each of the grouped z-step's 8 lanes per document reads 1, 2 or
// 4 consecutive words with one aligned load (the words past ceil(K / 32) are
// zero); 64 above 1024 topics, and above 2048 what the dense rows cover (16
// words for every 512 topics).
__host__ __device__ inline int bitmap_row_words(int K) {
    const int per_lane = (((K + 31) / 32) + 7) / 8;
    if (per_lane > 8) return 16 * ((K + 511) / 512);
    return 8 * (per_lane <= 1 ? 1 : per_lane <= 2 ? 2 : per_lane <= 4 ? 4 : 8);
}
// Dense rows of the z-step (zdense.cuh): a word's weights q as three planes of
// bytes, and a document's counts as planes of bytes in the same order.  Lane l
// of a warp owns the 4 NW consecutive topics [4 NW l, 4 NW l + 4 NW); a plane
// is 128 NW bytes.  Up to 512 topics a lane's bytes are consecutive; above,
// they lie in chunks of 16 bytes, chunk c of all lanes before chunk c + 1, so
// that a warp's 16-byte loads are consecutive and free of bank conflicts.
__host__ __device__ inline int dense_words(int K) {
    return K <= 128 ? 1 : K <= 256 ? 2 : K <= 512 ? 4 : 4 * ((K + 511) / 512);
}
__host__ __device__ inline int dense_row_bytes(int K) { return 3 * 128 * dense_words(K); }
__host__ __device__ inline int dense_pos(int K, int k) {
    if (K <= 512) return k;
    const int tpl = 4 * dense_words(K);
    const int l = k / tpl, b = k - l * tpl;
    return ((b >> 4) << 9) + (l << 4) + (b & 15);
}
// A document on a CTA of its own: a chain of warps up to here (zchain.cuh), all
// warps on each token above (zsplit.cuh).
constexpr int kChainMaxK = 8192;
// With documents of 2^16 tokens or more, whose counts take a second plane, the
// line lies here (one of 90,000 beside 500 others, ms per sweep, chain / split:
// K = 4,200 86 / 112, 6,000 103 / 112, 8,000 128 / 112).
constexpr int kChainWideMaxK = 6656;
// Warps per CTA of the warp-per-document z-step: the default and the largest
// accepted (the kernel's launch bounds are sized for it).
#ifndef PULDA_ZWARPS
#define PULDA_ZWARPS 4
#endif
constexpr int kZWarps = PULDA_ZWARPS;
// The batched (many-chain) z-step: the largest CTA in warps (its tuning
// candidates are the powers of two up to it) and the CTAs per SM its launch
// bounds ask for.
#ifndef PULDA_MULTI_WARPS
#define PULDA_MULTI_WARPS 8
#endif
#ifndef PULDA_MULTI_MINB
#define PULDA_MULTI_MINB 3
#endif
constexpr int kMultiWarps = PULDA_MULTI_WARPS;
// Words also keep their fixed-point weights q as dense rows, most frequent
// words first, up to this many bytes.  A word without a row is summed over its
// column (the same sums).
#ifndef PULDA_DENSE_BYTES
#define PULDA_DENSE_BYTES (2048ll << 20)
#endif
constexpr long long kDenseBytes = PULDA_DENSE_BYTES;

// Philox stream tags (counter word 3 = tag << 28 | aux).
enum : uint32_t { TAG_INIT = 1, TAG_POIS = 2, TAG_BETA = 3, TAG_REDRAW_POIS = 4, TAG_REDRAW_BETA = 5, TAG_Z = 6,
                  TAG_GAMMA = 7, TAG_GAMMA_BOOST = 8 };
// Dirichlet Phi-step (Algorithm 1): rows are summed in chunks of this many
// words, and a Gamma draw gives up after this many rejected attempts.
constexpr int kDirChunk = 256;
constexpr uint32_t kMaxGammaTry = 1u << 16;

// Slots of the per-sweep counter block on the device.
enum : int { ST_TOKENS = 0, ST_ABRANCH, ST_SUMMIN, ST_ZEROMASS, ST_DEADROWS, ST_NNZPHI, ST_ERROR, ST_SUMINT,
             ST_DOCSIDE, ST_COUNT = 12 };
// Running totals of the z-step slots live at ST_COUNT + slot and are cleared
// only at pulda_init.
constexpr int ST_TOTAL_SLOTS = 2 * ST_COUNT;
enum : unsigned long long { ERR_DEGENERATE = 1, ERR_INTERNAL = 2, ERR_GAMMA = 4, ERR_BOUNDS = 8, ERR_BARRIER = 16, ERR_COPY = 32 };

// Fixed tables of one beta, built on the host once.
struct HostTables {
    std::vector<uint32_t> thr;     // alias thresholds of every table, concatenated
    std::vector<uint16_t> alias;   // alias outcome, as an offset from the table's lo
    std::vector<int32_t> off;      // [kL+1] start of table t (t = 0: zero-truncated Pois(beta); t = l: Pois(beta+l))
    std::vector<int32_t> lo;       // [kL+1] smallest value of table t
    std::vector<int32_t> n;        // [kL+1] support size of table t
    std::vector<uint32_t> geo;     // [kGeoLen] P(gap <= g) * 2^32
    std::vector<double> gauss;     // [kGaussCells+1] inverse-normal nodes
};
int build_host_tables(float beta, HostTables *out);

// Device view of the same tables.
struct DevTables {
    const uint32_t *thr;
    const uint16_t *alias;
    const int32_t *off;
    const int32_t *lo;
    const int32_t *n;
    const uint32_t *geo;
    const double *gauss;
    double beta;
    const longlong2 *gauss_fix;    // [kGaussCells] lower node and width of the cells in units of 2^-58 (Dirichlet mode)
};

// Everything the Phi-step kernels read and write.
struct PhiArgs {
    int K, V;
    uint64_t seed;
    uint32_t sweep;
    const uint32_t *sweep_ptr;  // if set, the sweep counter is read here (graph replay)
    const int32_t *perm;        // [N] token ids grouped by word
    const int64_t *word_off;    // [V+1]
    const int32_t *word_order;  // [V] words by decreasing token count
    const int16_t *z;           // [N]
    DevTables tab;
    // staging: n columns at word_off, c columns at v*K (capacity K each)
    uint16_t *nst_k; uint32_t *nst_n; int32_t *nnz_n;
    uint16_t *cst_k; uint32_t *cst_c; int32_t *nnz_c;
    unsigned long long *S;      // [K] row sums S_k
    uint32_t *rowbuf;           // [V] scratch of the dead-row redraw
    int64_t *col_ptr;           // [V+1]
    // final per-word tables, at col_ptr
    uint16_t *topic; uint32_t *c; uint32_t *q; uint32_t *athr; uint16_t *atopic;
    // the alias slots packed as {threshold, column topic | alias topic << 16}
    // (written beside athr / atopic when set; the z-step then reads one 8-byte
    // slot per alias draw instead of a threshold and a topic)
    uint2 *apack;
    unsigned long long *A;      // [V]
    unsigned long long *vose_p; // [cap] scratch
    uint16_t *vose_stack;       // [cap] scratch
    uint32_t *bits;             // [V * KWp] nonzero-topic bits of each word's column
    int KW, KWp;
    uint8_t *qrow;              // dense rows of byte planes, dense_row_bytes(K) each
    const int32_t *row_slot;    // [V] the word's row in qrow, or -1
    int32_t *drow;              // [V] the same as the current Phi has it: -1 too where a q is 2^24 (25 bits)
    uint32_t *qdense;           // [V * K] q by topic (0 off the column): four documents per warp only, else null
    const float *alpha;         // [K]
    unsigned long long *rcp;    // [K] floor((2^127 - 1) / S_k), S_k shifted up to 64 bits (Polya urn)
    int *work, *work_warp;      // dynamic word counters: CTAs', warps'
    int n_big;                  // words (the first of word_order) that a CTA counts; the others a warp each
    unsigned long long *stats;  // [ST_COUNT]
    // words with more than heavy_word(N) tokens get their topic histogram from a
    // separate pass split over many CTAs
    const int32_t *heavy_row;   // [V] row of the word in heavy_hist, or -1
    uint32_t *heavy_hist;       // [n_heavy * K]
    int n_heavy;
    // Dirichlet Phi (Algorithm 1); gam is null for the Polya urn
    float *gam;                 // [V * K] Gamma draws, word-major
    double *Sd;                 // [K] row sums
    double *invS;               // [K] 1 / S_k (0 for an all-zero row)
    float *invSf;               // [K] 1 / S_k rounded to float (screening only)
    double *dpart;              // [ceil(V / kDirChunk) * K] chunk sums of the rows
    int counted;                // the n columns are already built (sort path): read them, do not histogram
};

// A word of a chain of N tokens with more tokens than heavy_word(N) is
// histogrammed in chunks of heavy_chunk(N) tokens by several CTAs before the
// per-word Phi-step pass.  The limit follows N: with 2^17 tokens for every N
// the largest words just below it were a tail that one CTA worked through
// alone (200 of the pass's 375 us with 12.4 M tokens).  At most 1,024 words
// are above it while N < 2^27, and fewer than N / 2^17 past that.
constexpr int64_t heavy_clamp(int64_t x, int64_t hi) { return x < 4096 ? 4096 : x > hi ? hi : x; }
constexpr int64_t heavy_word(int64_t N) { return heavy_clamp(N / 1024, int64_t(1) << 17); }
constexpr int64_t heavy_chunk_tokens(int64_t N) { return heavy_clamp(N / 2048, int64_t(1) << 16); }
// One chunk of a heavy word: chain, row in heavy_hist, word, token range.
struct HeavyChunk {
    int32_t chain, row, v, pad;
    int64_t begin, end;
};
void launch_heavy_hist(const PhiArgs *chains, const HeavyChunk *chunks, int n_chunks, int kmax, cudaStream_t st);
void launch_phi_tables_multi(const PhiArgs *chains, const int2 *items, int n_items, int kmax, cudaStream_t st);

struct ZArgs {
    const int64_t *doc_off;     // [D+1]
    const int32_t *doc_order;   // [D] documents by decreasing length
    int64_t D;
    const int32_t *w;           // [N]
    int16_t *z;                 // [N]
    const int64_t *col_ptr;
    const uint16_t *topic;
    const uint32_t *q;
    const unsigned long long *A;
    const uint32_t *athr;
    const uint16_t *atopic;
    const uint2 *apack;         // packed alias slots (PhiArgs::apack) or null: read athr / topic / atopic
    const uint32_t *bits;       // [V * KWp] nonzero-topic bits of each word's column
    const uint8_t *qrow;        // dense rows (PhiArgs::qrow) and each word's, or -1
    const int32_t *drow;
    const uint32_t *qdense;     // [V * K] q by topic: four documents per warp only
    // stale-count slices of long documents (k_z_step only): {row in m0, the
    // document, first token, tokens} is {y, x, z, w}; taken before the D documents
    const int4 *slices;
    int n_slices;
    const uint32_t *m0;         // [rows * K] pass-start counts of the sliced documents
    int K, KW, KWp;
    uint64_t seed;
    uint32_t sweep;
    const uint32_t *sweep_ptr;  // if set, the sweep counter is read here (graph replay)
    int64_t index_base;         // RNG index of token 0
    int path;                   // zstep_path: 0 auto, 1 a higher column limit, 2 the row wherever there is one
    int narrow;                 // 1: every document of the launch has fewer than 2^16 tokens (two count planes, else three)
    int *work;
    unsigned long long *stats;
};

// Launchers (kernels.cu).  All are asynchronous on `st`.
void launch_init_z(int64_t N, int K, uint64_t seed, int64_t index_base, int16_t *z, cudaStream_t st);
void launch_word_perm(int64_t N, int V, const int32_t *w, int64_t *word_off, int32_t *fill, int32_t *perm,
                      cudaStream_t st);
void launch_phi_counts(const PhiArgs &a, bool draw, int grid, cudaStream_t st);
void launch_phi_fixup(const PhiArgs &a, cudaStream_t st);
void launch_colptr_scan(const PhiArgs &a, cudaStream_t st);
void launch_phi_tables(const PhiArgs &a, cudaStream_t st);
void launch_z_step(const ZArgs &a, int warps_per_block, int grid, cudaStream_t st);
// The same with two documents per warp (zpair.cuh): K <= 1024 (else no CTA
// fits), documents of at most kNarrowMaxLen tokens, no slices.
void launch_z_step_pairs(const ZArgs &a, int warps_per_block, int grid, cudaStream_t st);
int z_pair_blocks_per_sm(int K, int warps_per_block);
// The documents doc_order[0 .. n_coop), one CTA each (zchain.cuh, zsplit.cuh);
// `wide`: one of them has more than kNarrowMaxLen tokens; `work` is a counter
// zeroed before the launch.
void launch_z_step_coop(const ZArgs &a, int n_coop, bool wide, int *work, int grid, cudaStream_t st);
int z_coop_blocks_per_sm(int K, bool wide);
// Automatic threshold of the long-document z-step: a document on one warp
// among 27 others on its SM takes about 1 us per token while the pass streams
// a token in 0.32 ns (K = 1000), so one longer than N / 3100 tokens would
// outlast the pass; the line lies a little below.  z-step ms at K = 1000,
// threshold 1,000 / 1,500 / 2,500 / none: N = 12.4M 4.93 / 4.62 / 4.18 / 7.14,
// N = 9.9M 4.04 / 3.85 / 3.48 / 6.02; K = 3000, N = 6.5M, threshold 500 /
// 1,000 / 2,000 / none: 8.88 / 6.90 / 7.27 / 16.1.
constexpr int64_t kCoopAutoDiv = 4500;
constexpr int64_t kCoopAutoDivPairs = 9000;     // two documents per warp: each takes twice as long
constexpr int64_t kCoopAutoMin = 256;
// The same over a batch's chains, whose passes are of mixed K (eight chains,
// 6.3M tokens, K 50 to 500: a sweep takes 3.97 ms at N / 8000, 4.35 at N /
// 4500, 4.68 at N / 2500).
constexpr int64_t kBatchCoopDiv = 8000;
// The same beside the grouped z-step, whose pass is faster and whose
// documents each advance more slowly (four share a warp's issue slots).
#ifndef PULDA_COOP_DIV_GROUPED
#define PULDA_COOP_DIV_GROUPED 16000
#endif
constexpr int64_t kCoopAutoDivGrouped = PULDA_COOP_DIV_GROUPED;
// Pass-start topic counts of the documents that the z-step takes in slices.
void launch_slice_counts(const int64_t *doc_off, const int32_t *sliced_docs, int n, const int16_t *z, int K,
                         uint32_t *m0, cudaStream_t st);
// Largest dynamic shared memory a CTA may opt in to (device attribute).
int smem_optin();
size_t z_step_smem(int K, int warps_per_block, bool narrow = false);
size_t phi_counts_smem(int K);
int64_t phi_warp_word_tokens();
int phi_big_words(int K, int64_t n, int64_t n_over, int grid);
void launch_doc_topic(const int64_t *doc_off, int64_t D, const int16_t *z, int K, int32_t *m_dk, cudaStream_t st);
void launch_n_dense(const PhiArgs &a, int32_t *n_kv, cudaStream_t st);
void launch_phi_values(const PhiArgs &a, float *phi, cudaStream_t st);
int z_step_blocks_per_sm(int K, int warps_per_block, bool narrow = false);
// Grouped z-step (zgroup.cu): 4 documents per warp, 8 lanes each, K <=
// kMaxKGrouped, documents of at most kMaxGroupDocLen tokens, every word with a
// dense q row; the warps of a CTA are z_groups_warps().
constexpr int kMaxGroupDocLen = 65535;
// A launch whose documents have at most this many tokens each keeps their counts
// in two planes (ZArgs::narrow; the CTA kernels: !wide).
constexpr int64_t kNarrowMaxLen = 65535;
// Length classes of documents (fold-in without allocation), eight to an octave
// and the longest first: those of 2^16 tokens or more, then those of at least
// coop_len (a CTA each, as the ones before), then the rest.  So the schedule is
// longest first, but for lengths within an eighth of each other or past 2^16; in
// any order within the three groups, a long document taken up late was the end
// of the pass (4,096 documents: 2.10 ms).  A class is in [0, kLengthClasses)
// whatever the length.
constexpr int kLengthKeys = 112;
constexpr int kLengthClasses = 1 + 2 * kLengthKeys;
__host__ __device__ inline int length_class(int64_t len, int64_t coop_len) {
    if (len > kNarrowMaxLen) return 0;
    const int n = len < 0 ? 0 : static_cast<int>(len);
    int e = 3;                                                   // n < 2^(e + 1), e >= 3
    while (n >> (e + 1)) ++e;
    const int key = n < 8 ? n : 8 * (e - 2) + ((n >> (e - 3)) & 7);       // at most 111
    return (len >= coop_len ? 1 : 1 + kLengthKeys) + kLengthKeys - 1 - key;
}
void launch_z_step_groups(const ZArgs &a, int grid, cudaStream_t st);
int z_groups_blocks_per_sm(int K);
int phi_counts_blocks_per_sm(int K);

// The count rebuild by sorting (countsort.cu): every token's key w K + z
// radix-sorted, runs of equal keys -> the n columns (nst_k, nst_n at
// word_off, nnz_n), bit-identical to the histogram pass's.  Needs V K < 2^32
// and count_sort_scratch_words(N) words of scratch.
size_t count_sort_scratch_words(int64_t N);
void launch_count_sort(const int32_t *w, const int16_t *z, int64_t N, int K, int V, const int64_t *word_off,
                       uint16_t *nst_k, uint32_t *nst_n, int32_t *nnz_n, uint32_t *scratch,
                       unsigned long long *stats, cudaStream_t st);

// Dirichlet Phi-step (dirichlet.cu), after the count-only pass has built the
// n columns: Gamma draws, row sums, and the kept entries staged in cst_k /
// cst_c (the draws' float bits) with nnz_c; the column scan and the table
// kernel follow as for the Polya urn.
void launch_dir_phi(const PhiArgs &a, cudaStream_t st);
size_t dir_part_count(int V, int K);

// Log-posterior diagnostic (diag.cu).  `counts` holds the n columns rebuilt
// from the current z (the count-only Phi-step pass); `scratch` is device
// memory of log_posterior_scratch_bytes(D, V, K) bytes whose first three
// doubles receive {total, document sum, topic sum}.
size_t log_posterior_scratch_bytes(int64_t D, int V, int K);
void launch_log_posterior(const int64_t *doc_off, int64_t D, const int16_t *z, int K, const float *alpha, double asum,
                          const PhiArgs &counts, double beta, bool symmetric, void *scratch, cudaStream_t st);

// The grid barrier of the one-launch batched sweep (device memory, zeroed).
struct GridBarrier {
    unsigned count;
    unsigned gen;
};

// The chains of one form of the z-step (dense_words up to 1,024 topics, one
// form to kChainMaxK and one above): their documents, n from `first` on in the form order,
// longest first: the first n_coop on CTAs, the others one per warp; the first
// n_wide have 2^16 tokens or more.
constexpr int kMaxForms = 6;
struct BatchForm {
    int kmax, first, n;
    int n_wide, n_coop;
    int z_grid, coop_grid;
};
constexpr int kBatchCounters = 2 + 3 * kMaxForms;     // work queues of a sweep

// One sweep of many chains: a launch or a few per phase, every kernel over all
// chains' work items (of a form, in the z-step), or one persistent launch for
// the Phi-step.  Pointers are device memory.
struct BatchLaunch {
    const HeavyChunk *heavy;     // heavy-word histogram chunks of every chain
    int n_heavy;
    const PhiArgs *phi;          // [n_chains], sweep_ptr = sweep
    const ZArgs *z;              // [n_chains], sweep_ptr = sweep
    int n_chains;
    const int2 *phi_items;       // (chain, word), most tokens first
    int n_phi_items, n_big;      // n_big: those counted by a CTA each
    int vmax;
    const int2 *form_items;      // (chain, document), form by form, longest first in each
    BatchForm form[kMaxForms];
    int n_forms;
    uint32_t *sweep;             // shared sweep counter, advanced by the first launch
    int *work;                   // [kBatchCounters] dynamic work queues
    int kmax;                    // largest K of the chains
    int phi_grid, z_warps;
    // streams beside the batch's for the z-step's launches, forked and joined
    // with the events
    cudaStream_t side[2 * kMaxForms - 1];
    cudaEvent_t ev_fork, ev_join[2 * kMaxForms - 1];
    // the one-launch form: its grid (all CTAs resident) and barrier
    int persist_grid;
    GridBarrier *bar;
    int table_stage;             // bytes of a warp's stage in its table phase (0: rows are written in place)
};
void launch_batch_sweep(const BatchLaunch &b, cudaStream_t st);
// The same sweep with the Phi-step as one cooperative launch; needs persist_grid <= SMs x
// batch_persistent_blocks_per_sm(kmax).
cudaError_t launch_batch_sweep_persistent(const BatchLaunch &b, cudaStream_t st);
int batch_persistent_blocks_per_sm(int kmax, bool narrow, int *table_stage);
// The grid barrier's self-test: `blocks` resident CTAs pass `rounds`
// barriers that expect blocks + missing arrivals.
cudaError_t launch_barrier_selftest(GridBarrier *bar, int blocks, int missing, int rounds, unsigned long long *err,
                                    unsigned *passed, cudaStream_t st);
int batch_phi_blocks_per_sm(int kmax);
int batch_z_blocks_per_sm(int kmax, int warps, bool narrow);
int batch_coop_blocks_per_sm(int kmax, bool wide);
// Documents on CTAs over (chain, document) items (coop.cu).
void launch_z_step_coop_multi(const ZArgs *chains, const int2 *items, int n_items, bool wide, int *work, int kmax, int grid,
                              cudaStream_t st);

// A request being folded in by the server (device slot table entry).
struct ServeSlot {
    int64_t off;          // first token in the arena
    int32_t len;          // tokens (>= 1)
    int32_t pos;          // next position of the current pass
    uint32_t sweep;       // current pass; 0 = initial topics not drawn yet
    uint32_t sweep_end;   // 1 + sweeps requested: done when sweep reaches it
    uint64_t seed;        // the request's Philox key
};
// Each active slot advances by up to `slice` tokens, one warp per slot; with
// window_ns > 0 also stopping at the first 32-token block boundary window_ns
// after the launch starts (every slot does at least one block).
// `narrow`: every active request of the launch has at most kNarrowMaxLen tokens.
void launch_serve_step(const ZArgs &a, ServeSlot *slots, const int32_t *active, int n_active, const int32_t *arena_w,
                       int16_t *arena_z, int64_t slice, int *work, int warps_per_block, int grid, uint64_t window_ns,
                       bool narrow, cudaStream_t st);
int serve_blocks_per_sm(int K, int warps_per_block);
// The same with one CTA per slot, for long requests; `wide`: one has more than
// kNarrowMaxLen tokens.
void launch_serve_step_coop(const ZArgs &a, ServeSlot *slots, const int32_t *active, int n_active, bool wide,
                            const int32_t *arena_w, int16_t *arena_z, int64_t slice, int *work, int grid,
                            uint64_t window_ns, cudaStream_t st);
int serve_coop_blocks_per_sm(int K, bool wide);
// With the handle's coop_min_len 0 (automatic), requests at least this long
// are served on CTAs, and all of them while a CTA is free for each.
constexpr int64_t kServeCoopAuto = 1024;

// What another translation unit needs to launch the z-step on a handle's
// current Phi (api.cpp).
struct HandleView {
    cudaStream_t stream;
    int device;      // the device the handle was created on
    int K, V;
    bool have_phi;
    int z_warps, z_grid;
    ZArgs zargs;     // Phi tables, K, path; corpus, RNG and scratch fields unset
};
}  // namespace pulda
struct pulda_handle;
namespace pulda {
bool handle_view(pulda_handle *h, HandleView *out);
int handle_fail(pulda_handle *h, int status, const char *msg);

}  // namespace pulda
