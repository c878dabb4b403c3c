// The batched variants of the sampling kernel (mcpd_pairs.cuh with BATCH): many instances of
// uneven size in one persistent launch, tables read through the read-only cache from per-instance
// descriptors.  Compiled for any degree (rows padded to eight entries, thresholds indexed by
// (n+, n-)) and, for coupled classes whose instances all have one uniform degree from 3 to 8,
// with that degree as a compile-time constant (mask-indexed thresholds up to degree 6), as the
// single-instance kernels are: degrees 3 and 6 here, 4, 5, 7 and 8 in mcpd_batch_deg.cu.  Separate
// translation units so that the library builds in parallel.
#include "mcpd_pairs.cuh"

namespace mcpd {

PairsKernelFn pick_batch(int coupled, int scan, int udeg) {
    if (coupled) {
        switch (udeg) {
            case 3: return pairs_kernel<true, false, true, 3>;
            case 6: return pairs_kernel<true, false, true, 6>;
            case 4: case 5: case 7: case 8: return pick_batch_degree(udeg);
            default: return pairs_kernel<true, false, true, 0>;
        }
    }
    return scan == MCPD_SCAN_SYSTEMATIC ? pairs_kernel<false, true, true, 0> : pairs_kernel<false, false, true, 0>;
}

int batch_kernel_degree(int coupled, int ext, int udeg) {
    (void)ext;                        // capped and lagged classes have the same builds
    return (coupled && udeg >= 3 && udeg <= 8) ? udeg : 0;
}

}  // namespace mcpd
