// The long-document z-step: one CTA per long document (corpus, fold-in, serving
// and batched forms), beside the one-warp kernel of kernels.cu that takes the
// rest.  The same draws, in the same order, so the topics are identical.
#include <algorithm>
#include <cstdint>

#include "device_rng.cuh"
#include "pulda_internal.h"
#include "zchain.cuh"
#include "zsplit.cuh"
#include "zstep.cuh"
#include "checks.cuh"

namespace pulda {
namespace {

// The CTA's next item from a shared counter.
__device__ __forceinline__ int next_item(CtaCtl &ctl, int *work) {
    __syncthreads();              // every thread has read the previous one
    if (threadIdx.x == 0) ctl.item = atomicAdd(work, 1);
    __syncthreads();
    return ctl.item;
}

// The forms: dense_words(K) up to 1,024 topics, 0 up to kChainMaxK, -1 above.
__host__ __forceinline__ int cta_form(int K) { return K > kChainMaxK ? -1 : z_nw(K); }
__host__ __forceinline__ int cta_threads(int K) { return K > kChainMaxK ? kSplitThreads : kChainThreads; }
__host__ __forceinline__ int cta_smem_bytes(int K) { return K > kChainMaxK ? split_smem_bytes(K) : chain_smem_bytes(K); }

// One document, by the CTA; false where its copies failed, and the CTA stops.
template <int NW>
__device__ __forceinline__ bool z_doc_cta(const ZArgs &a, uint8_t *sm, DocRun &r, uint32_t &phases) {
    if constexpr (NW < 0) {
        return z_doc_split(a, sm, r, phases);
    } else {
        z_doc_chain<NW>(a, sm, r, phases);
        return true;
    }
}

// The longest documents of a pass (dynamically scheduled, longest first):
// doc_order[0 .. n_coop).
template <int NW>
__global__ void __launch_bounds__(NW < 0 ? kSplitThreads : kChainThreads, NW < 0 ? 2 : 4) k_z_step_coop(ZArgs a, int n_coop, int *work) {
    extern __shared__ __align__(16) uint8_t csm[];
    CtaCtl &ctl = *reinterpret_cast<CtaCtl *>(csm);
    cta_begin(csm);
    uint32_t phases = 0;
    const uint32_t sweep = sweep_of(a);
    for (;;) {
        const int item = next_item(ctl, work);
        if (item >= n_coop) break;
        const int d = a.doc_order[item];
        const int64_t s = a.doc_off[d];
        const int len = static_cast<int>(a.doc_off[d + 1] - s);
        DocRun r{a.w + s, a.z + s, len, a.seed, a.index_base + s, sweep, 0, len, 1};
        if (!z_doc_cta<NW>(a, csm, r, phases)) break;
    }
    if (threadIdx.x < 32) flush_warp_counters(a.stats, ctl.cnt);
}

// Many chains of one form: their longest documents; items[0 .. n_items) are
// (chain, document) pairs.
template <int NW>
__global__ void __launch_bounds__(NW < 0 ? kSplitThreads : kChainThreads, NW < 0 ? 2 : 4) k_z_step_coop_multi(const ZArgs *chains, const int2 *items, int n_items,
                                                                        int *work) {
    extern __shared__ __align__(16) uint8_t csm[];
    CtaCtl &ctl = *reinterpret_cast<CtaCtl *>(csm);
    cta_begin(csm);
    uint32_t phases = 0;
    for (;;) {
        const int item = next_item(ctl, work);
        if (item >= n_items) break;
        const int2 it = items[item];
        const ZArgs a = chains[it.x];
        const int64_t s = a.doc_off[it.y];
        const int len = static_cast<int>(a.doc_off[it.y + 1] - s);
        DocRun r{a.w + s, a.z + s, len, a.seed, a.index_base + s, sweep_of(a), 0, len, 1};
        if (!z_doc_cta<NW>(a, csm, r, phases)) break;
        if (threadIdx.x < 32) flush_warp_counters(a.stats, ctl.cnt);
    }
}

// The long requests of a server: active[0 .. n_active) are their slots.
template <int NW>
__global__ void __launch_bounds__(NW < 0 ? kSplitThreads : kChainThreads, NW < 0 ? 2 : 4) k_serve_step_coop(ZArgs a, ServeSlot *slots, const int32_t *active,
                                                                   int n_active, const int32_t *arena_w,
                                                                   int16_t *arena_z, int64_t slice, int *work,
                                                                   uint64_t window_ns) {
    extern __shared__ __align__(16) uint8_t csm[];
    CtaCtl &ctl = *reinterpret_cast<CtaCtl *>(csm);
    cta_begin(csm);
    uint32_t phases = 0;
    for (;;) {
        const int item = next_item(ctl, work);
        if (item >= n_active) break;
        if (threadIdx.x == 0) ctl.deadline = window_ns ? global_ns() + window_ns : ~0ull;
        __syncthreads();
        const uint64_t deadline = ctl.deadline;
        const int idx = active[item];
        const ServeSlot sl = slots[idx];
        int16_t *z = arena_z + sl.off;
        uint32_t sweep = sl.sweep;
        int pos = sl.pos;
        if (sweep == 0) {
            for (int i = threadIdx.x; i < sl.len; i += blockDim.x) {
                const U4 u = draw(sl.seed, static_cast<uint32_t>(i), 0u, 0u, TAG_INIT, 0);
                z[i] = static_cast<int16_t>(__umulhi(u.x, static_cast<uint32_t>(a.K)));
            }
            __syncthreads();
            sweep = 1;
            pos = 0;
        }
        DocRun r{arena_w + sl.off, z, sl.len, sl.seed, 0, sweep, pos, slice,
                 static_cast<int>(sl.sweep_end - sweep), deadline};
        const bool ok = z_doc_cta<NW>(a, csm, r, phases);
        if (threadIdx.x == 0) {         // a request that failed is handed back, with the error
            slots[idx].sweep = ok ? r.sweep : sl.sweep_end;
            slots[idx].pos = r.pos;
        }
        if (!ok) break;
    }
    if (threadIdx.x < 32) flush_warp_counters(a.stats, ctl.cnt);
}

using CoopKernel = void (*)(ZArgs, int, int *);
CoopKernel coop_kernel(int K) {
    switch (cta_form(K)) {
        case 1: return k_z_step_coop<1>;
        case 2: return k_z_step_coop<2>;
        case 4: return k_z_step_coop<4>;
        case 8: return k_z_step_coop<8>;
        case 0: return k_z_step_coop<0>;
        default: return k_z_step_coop<-1>;
    }
}

using ServeCoopKernel = void (*)(ZArgs, ServeSlot *, const int32_t *, int, const int32_t *, int16_t *, int64_t, int *, uint64_t);
ServeCoopKernel serve_coop_kernel(int K) {
    switch (cta_form(K)) {
        case 1: return k_serve_step_coop<1>;
        case 2: return k_serve_step_coop<2>;
        case 4: return k_serve_step_coop<4>;
        case 8: return k_serve_step_coop<8>;
        case 0: return k_serve_step_coop<0>;
        default: return k_serve_step_coop<-1>;
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

int z_coop_blocks_per_sm(int K) { return blocks_per_sm(coop_kernel(K), cta_threads(K), cta_smem_bytes(K)); }

void launch_z_step_coop(const ZArgs &a, int n_coop, int *work, int grid, cudaStream_t st) {
    if (n_coop <= 0) return;
    coop_kernel(a.K)<<<std::max(1, std::min(grid, n_coop)), cta_threads(a.K), cta_smem_bytes(a.K), st>>>(a, n_coop, work);
}

using CoopMultiKernel = void (*)(const ZArgs *, const int2 *, int, int *);
static CoopMultiKernel coop_multi_kernel(int kmax) {
    switch (cta_form(kmax)) {
        case 1: return k_z_step_coop_multi<1>;
        case 2: return k_z_step_coop_multi<2>;
        case 4: return k_z_step_coop_multi<4>;
        case 8: return k_z_step_coop_multi<8>;
        case 0: return k_z_step_coop_multi<0>;
        default: return k_z_step_coop_multi<-1>;
    }
}
// Chains of one form need the shared memory of that form's largest K.
static int coop_multi_smem(int kmax) { return cta_form(kmax) == 0 ? chain_smem_bytes_upto(kmax) : cta_smem_bytes(kmax); }

int batch_coop_blocks_per_sm(int kmax) { return blocks_per_sm(coop_multi_kernel(kmax), cta_threads(kmax), coop_multi_smem(kmax)); }

void launch_z_step_coop_multi(const ZArgs *chains, const int2 *items, int n_items, int *work, int kmax, int grid,
                              cudaStream_t st) {
    if (n_items <= 0) return;
    coop_multi_kernel(kmax)<<<std::max(1, std::min(grid, n_items)), cta_threads(kmax), coop_multi_smem(kmax), st>>>(
        chains, items, n_items, work);
}

int serve_coop_blocks_per_sm(int K) { return blocks_per_sm(serve_coop_kernel(K), cta_threads(K), cta_smem_bytes(K)); }

void launch_serve_step_coop(const ZArgs &a, ServeSlot *slots, const int32_t *active, int n_active,
                            const int32_t *arena_w, int16_t *arena_z, int64_t slice, int *work, int grid,
                            uint64_t window_ns, cudaStream_t st) {
    if (n_active <= 0) return;
    cudaMemsetAsync(work, 0, sizeof(int), st);
    serve_coop_kernel(a.K)<<<std::max(1, std::min(grid, n_active)), cta_threads(a.K), cta_smem_bytes(a.K), st>>>(
        a, slots, active, n_active, arena_w, arena_z, slice, work, window_ns);
}

}  // namespace pulda
