// Batched sampling-kernel variants for coupled classes whose instances all have one uniform
// degree of 4, 5, 7 or 8 (degrees 3 and 6 are in mcpd_batch.cu): the degree is a compile-time
// constant (and, up to degree 6, thresholds are mask-indexed), as in the single-instance kernels.
// A separate translation unit so that the library builds in parallel.
#include "mcpd_pairs.cuh"

namespace mcpd {

PairsKernelFn pick_batch_degree(int udeg) {
    switch (udeg) {
        case 4: return pairs_kernel<true, false, true, 4>;
        case 5: return pairs_kernel<true, false, true, 5>;
        case 7: return pairs_kernel<true, false, true, 7>;
        case 8: return pairs_kernel<true, false, true, 8>;
        default: return nullptr;
    }
}

}  // namespace mcpd
