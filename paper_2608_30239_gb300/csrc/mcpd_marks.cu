// The sampling kernel with marks of the clones that a slot touches (mcpd_pairs.cuh with MARKS), for
// slots of few steps against their clones (mark_words): single instances here, batches in
// mcpd_batch_marks.cu.  Builds of their own: the same code switched off at run time cost coupled runs
// without marks 2 to 3% (333 clones, capped: 3.88 -> 4.00 ms; a lag of one sweep 17.9 -> 18.3 ms).
#include "mcpd_pairs.cuh"

namespace mcpd {

PairsKernelFn pick_marks(int coupled, int scan, bool batch, int udeg) {
    if (batch) return pick_batch_marks(coupled, scan, batch_kernel_degree(coupled, 0, udeg));
    if (coupled) {
        switch (udeg) {
            case 3: return pairs_kernel<true, false, false, 3, false, true>;
            case 4: return pairs_kernel<true, false, false, 4, false, true>;
            case 5: return pairs_kernel<true, false, false, 5, false, true>;
            case 6: return pairs_kernel<true, false, false, 6, false, true>;
            case 7: return pairs_kernel<true, false, false, 7, false, true>;
            case 8: return pairs_kernel<true, false, false, 8, false, true>;
            default: return pairs_kernel<true, false, false, 0, false, true>;
        }
    }
    if (scan == MCPD_SCAN_SYSTEMATIC) {
        switch (udeg) {
            case 3: return pairs_kernel<false, true, false, 3, false, true>;
            case 4: return pairs_kernel<false, true, false, 4, false, true>;
            case 5: return pairs_kernel<false, true, false, 5, false, true>;
            case 6: return pairs_kernel<false, true, false, 6, false, true>;
            default: return pairs_kernel<false, true, false, 0, false, true>;
        }
    }
    switch (udeg) {
        case 3: return pairs_kernel<false, false, false, 3, false, true>;
        case 4: return pairs_kernel<false, false, false, 4, false, true>;
        case 5: return pairs_kernel<false, false, false, 5, false, true>;
        case 6: return pairs_kernel<false, false, false, 6, false, true>;
        default: return pairs_kernel<false, false, false, 0, false, true>;
    }
}

}  // namespace mcpd
