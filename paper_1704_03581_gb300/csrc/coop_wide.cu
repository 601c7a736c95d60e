// The kernels with a CTA per document whose counts take three planes (2^16 tokens
// or more in a document), up to kChainMaxK topics: a translation unit of their
// own, compiled beside coop.cu.
#include "coop_kernels.cuh"

namespace pulda {

CtaKernels cta_kernels_wide(int form) {
    switch (form) {
        case 1: return cta_kernels<1, 3>();
        case 2: return cta_kernels<2, 3>();
        case 4: return cta_kernels<4, 3>();
        case 8: return cta_kernels<8, 3>();
        default: return cta_kernels<0, 3>();
    }
}

}  // namespace pulda
