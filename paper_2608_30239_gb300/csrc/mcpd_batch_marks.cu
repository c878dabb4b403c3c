// Batches of slots of few steps: the batched sampling kernel with marks (see mcpd_marks.cu).
#include "mcpd_pairs.cuh"

namespace mcpd {

PairsKernelFn pick_batch_marks(int coupled, int scan, int udeg) {
    if (coupled) {
        switch (udeg) {
            case 3: return pairs_kernel<true, false, true, 3, false, true>;
            case 4: return pairs_kernel<true, false, true, 4, false, true>;
            case 5: return pairs_kernel<true, false, true, 5, false, true>;
            case 6: return pairs_kernel<true, false, true, 6, false, true>;
            case 7: return pairs_kernel<true, false, true, 7, false, true>;
            case 8: return pairs_kernel<true, false, true, 8, false, true>;
            default: return pairs_kernel<true, false, true, 0, false, true>;
        }
    }
    return scan == MCPD_SCAN_SYSTEMATIC ? pairs_kernel<false, true, true, 0, false, true> : pairs_kernel<false, false, true, 0, false, true>;
}

}  // namespace mcpd
