// The kernels with a CTA per document: the corpus pass and fold-in, batched
// chains, the server.  NW: the form (cta_form); PL: planes of a document's counts
// up to kChainMaxK topics, two, or three (coop_wide.cu) in launches with a
// document of 2^16 tokens or more.
#pragma once
#include <cstdint>

#include "device_rng.cuh"
#include "pulda_internal.h"
#include "zchain.cuh"
#include "zsplit.cuh"
#include "zstep.cuh"
#include "checks.cuh"

namespace pulda {

using CoopKernel = void (*)(ZArgs, int, int *);
using CoopMultiKernel = void (*)(const ZArgs *, const int2 *, int, int *);
using ServeCoopKernel = void (*)(ZArgs, ServeSlot *, const int32_t *, int, const int32_t *, int16_t *, int64_t, int *, uint64_t);
struct CtaKernels {
    CoopKernel pass;
    CoopMultiKernel multi;
    ServeCoopKernel serve;
};

namespace {

// The CTA's next item from a shared counter.
__device__ __forceinline__ int next_item(CtaCtl &ctl, int *work) {
    __syncthreads();              // every thread has read the previous one
    if (threadIdx.x == 0) ctl.item = atomicAdd(work, 1);
    __syncthreads();
    return ctl.item;
}

// One document, by the CTA, its counts in PL planes.
template <int NW, int PL>
__device__ __forceinline__ void z_doc_cta(const ZArgs &a, uint8_t *sm, DocRun &r, uint32_t &phases) {
    if constexpr (NW < 0) z_doc_split(a, sm, r, phases);
    else z_doc_chain<NW, PL>(a, sm, r, phases);
}

// The longest documents of a pass (dynamically scheduled, longest first):
// doc_order[0 .. n_coop).
template <int NW, int PL>
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
        z_doc_cta<NW, PL>(a, csm, r, phases);
        if (ctl.failed) break;
    }
    if (threadIdx.x < 32) flush_warp_counters(a.stats, ctl.cnt);
}

// Many chains of one form: their longest documents; items[0 .. n_items) are
// (chain, document) pairs.
template <int NW, int PL>
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
        z_doc_cta<NW, PL>(a, csm, r, phases);
        if (ctl.failed) break;
        if (threadIdx.x < 32) flush_warp_counters(a.stats, ctl.cnt);
    }
}

// The long requests of a server: active[0 .. n_active) are their slots.
template <int NW, int PL>
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
        z_doc_cta<NW, PL>(a, csm, r, phases);
        if (threadIdx.x == 0) {         // a request that failed is handed back, with the error
            slots[idx].sweep = ctl.failed ? slots[idx].sweep_end : r.sweep;
            slots[idx].pos = r.pos;
        }
        if (ctl.failed) break;
    }
    if (threadIdx.x < 32) flush_warp_counters(a.stats, ctl.cnt);
}

template <int NW, int PL>
CtaKernels cta_kernels() { return {k_z_step_coop<NW, PL>, k_z_step_coop_multi<NW, PL>, k_serve_step_coop<NW, PL>}; }

}  // namespace

// The kernels of a form with three planes (coop_wide.cu); form >= 0.
CtaKernels cta_kernels_wide(int form);

}  // namespace pulda
