// CUDA kernels (sm_103a) for coupled score-weighted Markov chain pool decoding.
//
// pairs_kernel (mcpd_pairs.cuh): persistent; one block per SM (or several when the state is small); every
// warp takes chunks of slots and runs each slot's coupled pairs (Algorithm 3) to their meetings, two
// lanes to a pair, and then its single chains, a lane each, under the fixed horizon B with slot
// refill (Algorithm 4).  Per lane, shared memory holds one chain's clone bit set and its
// per-pool positive counts (one byte each), laid out word-interleaved over the warp's 32 lanes so
// that the per-step loads of different lanes never share a bank.  The clone->pool rows, the alias
// table of the scan weights and the acceptance thresholds are staged once per block.  The hot loop is integer-only: a Philox4x32-10 block
// feeds two steps, the site comes from the alias table, the full conditional from a table lookup
// indexed by (n+, n-), and the update from a 64-bit integer comparison.  The estimator
// H_{k:l} is accumulated exactly in integers, only when a site flips (see the head of mcpd_pairs.cuh), and
// slot sums go to N*_p buckets with 64/128-bit integer atomics, so the result does not depend on
// the schedule.
#include <cuda_runtime.h>
#include <stdint.h>

#include "mcpd_device.cuh"
#include "mcpd_internal.h"
#include "mcpd_pairs.cuh"

namespace mcpd {
namespace {

// theta_j = (sum_{n ascending} S1[n][j] / n) / (P L);  Q_j = (sum_n S2[n][j] / n^2) / L^2;
// se_j = sqrt(max(0, (Q_j - (P theta_j) theta_j) / (P (P - 1)))).  Every operation is an
// explicitly rounded IEEE double operation, in this order.
__device__ __forceinline__ void finalize_one(const unsigned long long *S1, const unsigned long long *S2lo,
                                             const unsigned long long *S2hi, int na, int nb, long long P,
                                             long long L, int j, double *est, double *se) {
    const double dP = static_cast<double>(P), dL = static_cast<double>(L);
    double s1 = 0.0, s2 = 0.0;
    for (int b = 0; b < nb; ++b) {
        const size_t idx = static_cast<size_t>(b) * na + j;
        const double n = static_cast<double>(b + 1);
        s1 = __dadd_rn(s1, __ddiv_rn(static_cast<double>(static_cast<long long>(S1[idx])), n));
        const double sq = __dadd_rn(__dmul_rn(static_cast<double>(S2hi[idx]), 18446744073709551616.0),
                                    static_cast<double>(S2lo[idx]));
        s2 = __dadd_rn(s2, __ddiv_rn(sq, __dmul_rn(n, n)));
    }
    const double th = __ddiv_rn(s1, __dmul_rn(dP, dL));
    *est = th;
    if (P < 2) { *se = __longlong_as_double(0x7FF8000000000000LL); return; }
    const double Q = __ddiv_rn(s2, __dmul_rn(dL, dL));
    const double var = __ddiv_rn(__dsub_rn(Q, __dmul_rn(__dmul_rn(dP, th), th)),
                                 __dmul_rn(dP, __dsub_rn(dP, 1.0)));
    *se = var > 0.0 ? __dsqrt_rn(var) : 0.0;
}

__global__ void finalize_kernel(const unsigned long long *S1, const unsigned long long *S2lo,
                                const unsigned long long *S2hi, int na, int nb, long long P,
                                long long L, double *est, double *se) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= na) return;
    finalize_one(S1, S2lo, S2hi, na, nb, P, L, j, &est[j], &se[j]);
}

// Batched finalize: one thread per (instance, clone), outputs concatenated in instance order.
__global__ void finalize_batch_kernel(const InstDesc *insts, const int32_t *clone_inst,
                                      const int32_t *clone_local, long long total, double *est,
                                      double *se) {
    const long long g = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (g >= total) return;
    const InstDesc &d = insts[clone_inst[g]];
    finalize_one(d.S1, d.S2lo, d.S2hi, d.na, d.nb, d.P_total, d.L, clone_local[g], &est[g], &se[g]);
}

__global__ void philox_kernel(const uint32_t *ctr, uint32_t k0, uint32_t k1, uint32_t *out, long long n) {
    const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
    const uint4 o = philox10(c, k0, k1);
    out[4 * i] = o.x; out[4 * i + 1] = o.y; out[4 * i + 2] = o.z; out[4 * i + 3] = o.w;
}

using PairsFn = PairsKernelFn;

PairsFn pick(int coupled, int scan, bool batch, int udeg, bool marks) {
    if (marks) return pick_marks(coupled, scan, batch, udeg);
    if (batch) return pick_batch(coupled, scan, batch_kernel_degree(coupled, 0, udeg));
    if (coupled) {
        switch (udeg) {
            case 3: return pairs_kernel<true, false, false, 3>;
            case 4: return pairs_kernel<true, false, false, 4>;
            case 5: return pairs_kernel<true, false, false, 5>;
            case 6: return pairs_kernel<true, false, false, 6>;
            case 7: return pairs_kernel<true, false, false, 7>;
            case 8: return pairs_kernel<true, false, false, 8>;
            default: return pairs_kernel<true, false, false, 0>;
        }
    }
    if (scan == MCPD_SCAN_SYSTEMATIC) {
        switch (udeg) {
            case 3: return pairs_kernel<false, true, false, 3>;
            case 4: return pairs_kernel<false, true, false, 4>;
            case 5: return pairs_kernel<false, true, false, 5>;
            case 6: return pairs_kernel<false, true, false, 6>;
            default: return pairs_kernel<false, true, false, 0>;
        }
    }
    switch (udeg) {
        case 3: return pairs_kernel<false, false, false, 3>;
        case 4: return pairs_kernel<false, false, false, 4>;
        case 5: return pairs_kernel<false, false, false, 5>;
        case 6: return pairs_kernel<false, false, false, 6>;
        default: return pairs_kernel<false, false, false, 0>;
    }
}

int max_warps(int coupled, int scan, int udeg, bool batch, bool marks) {
    cudaFuncAttributes a{};
    if (cudaFuncGetAttributes(&a, pick(coupled, scan, batch, udeg, marks)) != cudaSuccess) return 16;
    return a.maxThreadsPerBlock / 32;
}

}  // namespace

int pairs_max_smem(int device, size_t *bytes) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess)
        return MCPD_ECUDA;
    *bytes = static_cast<size_t>(v);
    return MCPD_OK;
}

int launch_pairs(const KParams &kp, int grid, int block, size_t smem, void *stream) {
    if (kp.trace_rec) return launch_pairs_trace(kp, grid, block, smem, stream);
    const BParams none{};
    pick(kp.coupled, kp.scan, false, kp.udeg, kp.marks > 0)<<<grid, block, smem, static_cast<cudaStream_t>(stream)>>>(kp, none);
    return cudaGetLastError() == cudaSuccess ? MCPD_OK : MCPD_ECUDA;
}

int launch_batch(const BParams &bp, int grid, int block, size_t smem, void *stream) {
    const KParams none{};
    pick(bp.coupled, bp.scan, true, bp.udeg, bp.marks > 0)<<<grid, block, smem, static_cast<cudaStream_t>(stream)>>>(none, bp);
    return cudaGetLastError() == cudaSuccess ? MCPD_OK : MCPD_ECUDA;
}

int launch_finalize_batch(const InstDesc *insts, int n_inst, const int32_t *clone_inst,
                          const int32_t *clone_local, long long total_clones, double *est,
                          double *se, void *stream) {
    (void)n_inst;
    if (total_clones <= 0) return MCPD_OK;
    finalize_batch_kernel<<<static_cast<unsigned>((total_clones + 127) / 128), 128, 0, static_cast<cudaStream_t>(stream)>>>(
        insts, clone_inst, clone_local, total_clones, est, se);
    return cudaGetLastError() == cudaSuccess ? MCPD_OK : MCPD_ECUDA;
}

int launch_finalize(const unsigned long long *S1, const unsigned long long *S2lo,
                    const unsigned long long *S2hi, int na, int nb, long long P, long long L,
                    double *est, double *se, void *stream) {
    finalize_kernel<<<(na + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(S1, S2lo, S2hi, na, nb, P, L, est, se);
    return cudaGetLastError() == cudaSuccess ? MCPD_OK : MCPD_ECUDA;
}

int launch_philox(const uint32_t *ctr, uint32_t k0, uint32_t k1, uint32_t *out, long long n, void *stream) {
    if (n <= 0) return MCPD_OK;
    philox_kernel<<<static_cast<unsigned>((n + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(ctr, k0, k1, out, n);
    return cudaGetLastError() == cudaSuccess ? MCPD_OK : MCPD_ECUDA;
}

int pairs_shape(int coupled, int scan, int udeg, bool batch, size_t tables, int wpp, size_t smem_optin,
                long long P, int sm_count, int warps, bool, bool marks, PairsShape *out) {
    const int cap = max_warps(coupled, scan, udeg, batch, marks);
    auto bytes = [&](int w) { return pairs_smem_bytes(tables, wpp, w); };
    auto most = [&](size_t budget) {
        int best = 0;
        for (int w = 1; w <= cap && bytes(w) <= budget; ++w) best = w;
        return best;
    };
    auto resident = [&](int w, int *per_sm) {
        *per_sm = 1;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, pick(coupled, scan, batch, udeg, marks), w * 32,
                                                             bytes(w)) == cudaSuccess;
    };
    // The limit of the interface: the tables and, coupled, both chains of one warp's pairs.
    if (bytes(coupled ? 2 : 1) > smem_optin) return MCPD_ETOO_LARGE;
    int w1 = most(smem_optin);
    // The attribute is a permission shared by every launch of the kernel (the classes of a batch
    // have different sizes): allow the device's opt-in maximum.
    if (cudaFuncSetAttribute(pick(coupled, scan, batch, udeg, marks), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem_optin)) != cudaSuccess)
        return MCPD_ECUDA;
    PairsShape s;
    if (warps > 0) {
        if (warps > w1) return MCPD_EINVAL;
        s.warps = warps;
        if (!resident(warps, &s.per_sm)) return MCPD_ECUDA;
    } else {
        s.warps = w1;
        if (!resident(w1, &s.per_sm)) return MCPD_ECUDA;
        if (!batch) {
            // Two blocks per SM (each with its own copy of the tables) when that holds more warps.
            const int w2 = most(smem_optin / 2);
            int per2 = 1;
            if (w2 >= 1 && resident(w2, &per2) && per2 * w2 > s.per_sm * s.warps) { s.warps = w2; s.per_sm = per2; }
            if (P > 0) s.warps = chunk_shape(P, static_cast<long long>(sm_count) * s.per_sm, s.warps, kBank).warps;
        }
    }
    s.smem = bytes(s.warps);
    if (s.per_sm < 1) s.per_sm = 1;
    *out = s;
    return MCPD_OK;
}

}  // namespace mcpd
