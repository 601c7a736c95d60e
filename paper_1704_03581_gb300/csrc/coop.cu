// The long-document z-step: one CTA per long document (corpus, fold-in, serving
// and batched forms), beside the one-warp kernel of kernels.cu that takes the
// rest.  The same draws, in the same order, so the topics are identical.
#include <algorithm>
#include <cstdint>

#include "coop_kernels.cuh"

namespace pulda {
namespace {

// The forms: dense_words(K) up to 1,024 topics, 0 up to kChainMaxK, -1 above
// (there any document's counts have three planes).
bool split(int K, bool wide) { return K > (wide ? kChainWideMaxK : kChainMaxK); }
int cta_form(int K, bool wide) { return split(K, wide) ? -1 : z_nw(K); }
int cta_threads(int K, bool wide) { return split(K, wide) ? kSplitThreads : kChainThreads; }
int cta_smem_bytes(int K, bool wide) { return split(K, wide) ? split_smem_bytes(K) : chain_smem_bytes(K, wide ? 3 : 2); }
// Chains of one form need the shared memory of that form's largest K.
int multi_smem_bytes(int kmax, bool wide) {
    return cta_form(kmax, wide) == 0 ? chain_smem_bytes_upto(kmax, wide ? 3 : 2) : cta_smem_bytes(kmax, wide);
}

CtaKernels kernels_of(int K, bool wide) {
    const int form = cta_form(K, wide);
    if (wide && form >= 0) return cta_kernels_wide(form);
    switch (form) {
        case 1: return cta_kernels<1, 2>();
        case 2: return cta_kernels<2, 2>();
        case 4: return cta_kernels<4, 2>();
        case 8: return cta_kernels<8, 2>();
        case 0: return cta_kernels<0, 2>();
        default: return cta_kernels<-1, 2>();
    }
}

template <typename F>
int blocks_per_sm(F *kern, int threads, size_t smem) {
    allow_dynamic_smem(kern);
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, threads, smem);
    return b > 0 ? b : 1;
}

}  // namespace

int z_coop_blocks_per_sm(int K, bool wide) { return blocks_per_sm(kernels_of(K, wide).pass, cta_threads(K, wide), cta_smem_bytes(K, wide)); }

void launch_z_step_coop(const ZArgs &a, int n_coop, bool wide, int *work, int grid, cudaStream_t st) {
    if (n_coop <= 0) return;
    kernels_of(a.K, wide).pass<<<std::max(1, std::min(grid, n_coop)), cta_threads(a.K, wide), cta_smem_bytes(a.K, wide), st>>>(a, n_coop, work);
}

int batch_coop_blocks_per_sm(int kmax, bool wide) {
    return blocks_per_sm(kernels_of(kmax, wide).multi, cta_threads(kmax, wide), multi_smem_bytes(kmax, wide));
}

void launch_z_step_coop_multi(const ZArgs *chains, const int2 *items, int n_items, bool wide, int *work, int kmax, int grid,
                              cudaStream_t st) {
    if (n_items <= 0) return;
    kernels_of(kmax, wide).multi<<<std::max(1, std::min(grid, n_items)), cta_threads(kmax, wide), multi_smem_bytes(kmax, wide), st>>>(
        chains, items, n_items, work);
}

int serve_coop_blocks_per_sm(int K, bool wide) { return blocks_per_sm(kernels_of(K, wide).serve, cta_threads(K, wide), cta_smem_bytes(K, wide)); }

void launch_serve_step_coop(const ZArgs &a, ServeSlot *slots, const int32_t *active, int n_active, bool wide,
                            const int32_t *arena_w, int16_t *arena_z, int64_t slice, int *work, int grid,
                            uint64_t window_ns, cudaStream_t st) {
    if (n_active <= 0) return;
    cudaMemsetAsync(work, 0, sizeof(int), st);
    kernels_of(a.K, wide).serve<<<std::max(1, std::min(grid, n_active)), cta_threads(a.K, wide), cta_smem_bytes(a.K, wide), st>>>(
        a, slots, active, n_active, arena_w, arena_z, slice, work, window_ns);
}

}  // namespace pulda
