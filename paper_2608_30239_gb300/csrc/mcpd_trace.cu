// The recording variants of the sampling kernel: the single-instance kernel (mcpd_pairs.cuh),
// coupled and uncoupled, compiled with TRACE, which also writes, for the first replications of every
// traced slot, the meeting time, the completion time and per draw the site and which chains flipped
// (MCPD_FETCH_TRACE_REC).  They
// exist for the trajectory parity tests against the CPU oracle; a plan launches them only when
// params.trace_steps > 0, and the production variants compile none of the recording.  A separate
// translation unit so that the library builds in parallel.
#include "mcpd_pairs.cuh"

namespace mcpd {
namespace {

using TraceFn = void (*)(const KParams, const BParams);

TraceFn pick_trace(int coupled, int scan, int udeg) {
    if (!coupled && scan == MCPD_SCAN_SYSTEMATIC) {
        switch (udeg) {
            case 3: return pairs_kernel<false, true, false, 3, true>;
            case 4: return pairs_kernel<false, true, false, 4, true>;
            case 5: return pairs_kernel<false, true, false, 5, true>;
            case 6: return pairs_kernel<false, true, false, 6, true>;
            default: return pairs_kernel<false, true, false, 0, true>;
        }
    }
    if (!coupled) {
        switch (udeg) {
            case 3: return pairs_kernel<false, false, false, 3, true>;
            case 4: return pairs_kernel<false, false, false, 4, true>;
            case 5: return pairs_kernel<false, false, false, 5, true>;
            case 6: return pairs_kernel<false, false, false, 6, true>;
            default: return pairs_kernel<false, false, false, 0, true>;
        }
    }
    switch (udeg) {
        case 3: return pairs_kernel<true, false, false, 3, true>;
        case 4: return pairs_kernel<true, false, false, 4, true>;
        case 5: return pairs_kernel<true, false, false, 5, true>;
        case 6: return pairs_kernel<true, false, false, 6, true>;
        case 7: return pairs_kernel<true, false, false, 7, true>;
        case 8: return pairs_kernel<true, false, false, 8, true>;
        default: return pairs_kernel<true, false, false, 0, true>;
    }
}

}  // namespace

int launch_pairs_trace(const KParams &kp, int grid, int block, size_t smem, void *stream) {
    if (!kp.trace_rec || kp.trace_stride <= 0) return MCPD_EINVAL;
    const BParams none{};
    if (cudaFuncSetAttribute(pick_trace(kp.coupled, kp.scan, kp.udeg), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem)) != cudaSuccess)
        return MCPD_ECUDA;
    pick_trace(kp.coupled, kp.scan, kp.udeg)<<<grid, block, smem, static_cast<cudaStream_t>(stream)>>>(kp, none);
    return cudaGetLastError() == cudaSuccess ? MCPD_OK : MCPD_ECUDA;
}

}  // namespace mcpd
