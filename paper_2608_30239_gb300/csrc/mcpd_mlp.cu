// Learned scan weights and initial marginals: per-clone features, a 16-64-64-2 MLP with bf16
// parameters and fp32 accumulation, its loss, backward pass and Adam update, and the two heads.
//
// Not in the paper.  The paper proves that any fixed positive scan weights leave pi invariant
// (Proposition 1) and that the coupled estimator is unbiased from any initial distribution
// (Theorem 1), so scan weights w and initial marginals nu predicted from the observed design are
// admissible inputs of the method: w = (1 - a) softmax(o_1) + a / n (a = 0.5 keeps every site's
// weight >= 0.5 / n) and nu = clamp(sigmoid(o_2), 1e-6, 1 - 1e-6).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "mcpd_internal.h"

namespace mcpd {
namespace {

constexpr int F = 16, H = 64, O = 2;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + H * F, OFF_W2 = OFF_B1 + H, OFF_B2 = OFF_W2 + H * H;
constexpr int OFF_W3 = OFF_B2 + H, OFF_B3 = OFF_W3 + O * H, NPARAM = OFF_B3 + O;   // 5378

// The row kernels work tiles of 64 rows per block of 256 threads.  Activations lie in shared memory
// feature-major, [feature][row] with rows padded to 68 floats: a thread owns 4 rows x 4 features of a
// layer and reads both factors of 16 multiply-adds with two 16-byte loads, and the gradient's
// products read 4 rows of a feature with one (68 = 4 mod 32, so 8 lanes reading 16 bytes of 8
// features hit 32 banks).  Bound by the FP32 pipe and shared memory; every sum over features runs
// in feature order.  (One thread per row, with its activations in local memory and two scalar
// loads per multiply-add of the gradient, took 46 us forward and 2.3 ms backward for 83,072 rows.)
constexpr int TR = 64, LD = TR + 4, TB = 256;
constexpr int SW1 = 0, SB1 = SW1 + F * H, SW2 = SB1 + H, SB2 = SW2 + H * H, SW3 = SB2 + H, SB3 = SW3 + O * H,
              SPARAM = (SB3 + O + 3) / 4 * 4;                    // floats; W1 and W2 stored [in][out]

// Parameters to shared memory in fp32, W1 and W2 transposed to [in][out].  A thread loads 8 inputs of an
// output, a warp 32 outputs of them, so that the transposed stores are conflict-free and all loads are
// in flight at once, and rows one tile ahead (one parameter at a time, in the order of W, and rows when
// their tile comes: 50 rows 10.8 us forward and 20.6 backward against 7.8 and 16.5, 83,072 rows 37.0 and 94.3
// against 29.7 and 89.2).
__device__ __forceinline__ void load8(const __nv_bfloat16 *W, bool wide, float (&v)[8]) {
    if (wide) {
        const uint4 q = __ldg(reinterpret_cast<const uint4 *>(W));
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            v[2 * u] = __uint_as_float(w[u] << 16);
            v[2 * u + 1] = __uint_as_float(w[u] & 0xFFFF0000u);
        }
    } else {                              // the caller's array need only hold bf16
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __bfloat162float(W[u]);
    }
}
__device__ __forceinline__ void stage_params(const __nv_bfloat16 *W, float *sW) {
    static_assert(OFF_W1 % 8 == 0 && OFF_W2 % 8 == 0 && H * F / 8 <= TB && H * H / 8 == 2 * TB, "load8 per thread");
    const bool wide = (reinterpret_cast<uintptr_t>(W) & 15u) == 0;
    const int t = threadIdx.x, out = t % H, in = t / H * 8;
    float a[8], b[8], c[8] = {};
    load8(W + OFF_W2 + out * H + in, wide, a);
    load8(W + OFF_W2 + out * H + in + TB / H * 8, wide, b);
    if (t < H * F / 8) load8(W + OFF_W1 + out * F + in, wide, c);
    const float b1 = __bfloat162float(W[OFF_B1 + t % H]), rest = __bfloat162float(W[OFF_B2 + min(t, NPARAM - OFF_B2 - 1)]);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        sW[SW2 + (in + u) * H + out] = a[u];
        sW[SW2 + (in + TB / H * 8 + u) * H + out] = b[u];
        if (t < H * F / 8) sW[SW1 + (in + u) * H + out] = c[u];
    }
    if (t < H) sW[SB1 + t] = b1;
    if (t < NPARAM - OFF_B2) sW[SB2 + t] = rest;
}

// Rows r0 .. r0 + 63 of X to sX [feature][row]; zeros past n.  A thread holds 4 features of a row, loaded
// while the tile before is worked.
__device__ __forceinline__ float4 load_rows(long long n, long long r0, const float *X, bool wide) {
    const long long r = r0 + threadIdx.x / 4;
    const float *const p = X + r * F + threadIdx.x % 4 * 4;
    if (r >= n) return make_float4(0.f, 0.f, 0.f, 0.f);
    if (wide) return *reinterpret_cast<const float4 *>(p);
    return make_float4(p[0], p[1], p[2], p[3]);
}
__device__ __forceinline__ void stage_rows(const float4 &v, float *sX) {
    static_assert(TR * F == 4 * TB, "four values per thread");
    float *const at = sX + threadIdx.x % 4 * 4 * LD + threadIdx.x / 4;
    at[0] = v.x; at[LD] = v.y; at[2 * LD] = v.z; at[3 * LD] = v.w;
}

// Two fp32 values in a register pair; fma2 is an fmaf of each (one instruction issues both).  The gradient's
// products pair rows, the layers' outputs: backward 98.5 -> 94.3 us for 83,072 rows, 4.70 -> 4.28 ms for 5e6.
using f2 = unsigned long long;
__device__ __forceinline__ f2 pack(float x, float y) {
    f2 v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
    return v;
}
__device__ __forceinline__ float2 unpack(f2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// acc[i][j] = bias[c0 + j] + sum_k A[k][r0 + i] B[k][c0 + j], k ascending.
template <int K>
__device__ __forceinline__ void tile_gemm(const float *A, const float *B, const float *bias, int r0, int c0, float (&acc)[4][4]) {
    f2 sum[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) sum[i][j] = bias ? pack(bias[c0 + 2 * j], bias[c0 + 2 * j + 1]) : 0ull;
#pragma unroll 8
    for (int k = 0; k < K; ++k) {
        const float4 a = *reinterpret_cast<const float4 *>(A + k * LD + r0);
        const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(B + k * H + c0);
        const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const f2 ai = pack(av[i], av[i]);
            sum[i][0] = fma2(b.x, ai, sum[i][0]);
            sum[i][1] = fma2(b.y, ai, sum[i][1]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float2 v = unpack(sum[i][j]);
            acc[i][2 * j] = v.x;
            acc[i][2 * j + 1] = v.y;
        }
}
// out[c0 + j][r0 + i] = f(acc[i][j])
template <typename Fn>
__device__ __forceinline__ void tile_store(float *out, int r0, int c0, const float (&acc)[4][4], Fn f) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
        *reinterpret_cast<float4 *>(out + (c0 + j) * LD + r0) =
            make_float4(f(acc[0][j], 0, j), f(acc[1][j], 1, j), f(acc[2][j], 2, j), f(acc[3][j], 3, j));
}

// A thread's place in a 16 x 16 grid of 4 x 4 blocks: a warp takes 8 by 4 of them, so that a 16-byte load or
// store of 8 lanes is one run of 128 bytes along the fast side and 4 addresses along the other.  (A warp of
// 16 by 2 took 3 wavefronts for the two loads of a product against 2, and its stores conflicted 4-fold: 83,072
// rows 29.7 us forward and 88.2 backward against 26.6 and 82.0.)
__device__ __forceinline__ int fast_side() { return (threadIdx.x & 7) + (threadIdx.x >> 5 & 1) * 8; }
__device__ __forceinline__ int slow_side() { return (threadIdx.x >> 3 & 3) + (threadIdx.x >> 6) * 4; }

constexpr int FWD_SMEM = (SPARAM + (F + 2 * H) * LD) * 4;

// H1 = relu(W1 x + b1), H2 = relu(W2 H1 + b2), out = W3 H2 + b3.
__global__ void __launch_bounds__(TB) mlp_forward_kernel(long long n, const float *X, const __nv_bfloat16 *W, float *Out) {
    extern __shared__ __align__(16) float sm[];
    float *sW = sm, *sX = sW + SPARAM, *sH1 = sX + F * LD, *sH2 = sH1 + H * LD;
    stage_params(W, sW);
    const int c0 = slow_side() * 4, r0 = fast_side() * 4;
    const auto relu = [](float v, int, int) { return fmaxf(v, 0.f); };
    const bool wide = (reinterpret_cast<uintptr_t>(X) & 15u) == 0;
    const long long first = static_cast<long long>(blockIdx.x) * TR, stride = static_cast<long long>(gridDim.x) * TR;
    float4 x = load_rows(n, first, X, wide);
    for (long long row = first; row < n; row += stride) {
        __syncthreads();
        stage_rows(x, sX);
        x = load_rows(n, row + stride, X, wide);
        __syncthreads();
        float acc[4][4];
        tile_gemm<F>(sX, sW + SW1, sW + SB1, r0, c0, acc);
        tile_store(sH1, r0, c0, acc, relu);
        __syncthreads();
        tile_gemm<H>(sH1, sW + SW2, sW + SB2, r0, c0, acc);
        tile_store(sH2, r0, c0, acc, relu);
        __syncthreads();
        if (threadIdx.x < TR * O) {
            const int r = threadIdx.x % TR, o = threadIdx.x / TR;
            float v = sW[SB3 + o];
#pragma unroll 16
            for (int b = 0; b < H; ++b) v = fmaf(sW[SW3 + o * H + b], sH2[b * LD + r], v);
            if (row + r < n) Out[(row + r) * O + o] = v;
        }
    }
}

// Chunks of rows of the parameter gradient: two blocks on each of 152 SMs when the rows allow it, at most
// 1024 rows each (the length of one fp32 sum), whole tiles.  The first chunks take a tile more where they
// do not divide (equal chunks, 260 of 5 tiles, left 44 SMs with one block of 83,072 rows: 82.0 against 73.8 us).
// A function of the row count alone, so the sum is reproducible.
constexpr int BLOCKS = 304, TILES = 1024 / TR;
long long tiles_of(long long n) { return (n + TR - 1) / TR; }
long long chunks_of(long long n) {
    const long long tiles = tiles_of(n);
    return tiles <= BLOCKS ? tiles : (tiles <= BLOCKS * TILES ? BLOCKS : (tiles + TILES - 1) / TILES);
}

constexpr int BWD_SMEM = (SPARAM + H * H + (F + 4 * H) * LD + 2 * TR) * 4;

// Partial parameter gradients of one chunk of rows: the activations recomputed, dOut back-propagated
// to dZ2 and dZ1, and gW1 = dZ1^T X, gb1 = sum dZ1, gW2 = dZ2^T H1, gb2 = sum dZ2, gW3 = dOut^T H2,
// gb3 = sum dOut summed over the chunk's rows in registers, in row order (gW1 and gW2 the even and the
// odd rows apart); nothing per row goes to
// memory.  A thread owns 16 entries of gW2 and 4 of gW1 (features 16 apart: conflict-free loads), and
// one of gb1, gb2 or gW3; two warps take gb3.
__global__ void __launch_bounds__(TB) mlp_backward_kernel(long long n, long long tiles, const float *X, const __nv_bfloat16 *W,
                                                          const float *dOut, float *partials) {
    extern __shared__ __align__(16) float sm[];
    float *sW = sm, *sW2 = sW + SPARAM, *sX = sW2 + H * H, *sH1 = sX + F * LD, *sH2 = sH1 + H * LD,
          *sD2 = sH2 + H * LD, *sD1 = sD2 + H * LD, *sO = sD1 + H * LD;
    stage_params(W, sW);
    {
        float v[H * H / TB];
#pragma unroll
        for (int i = 0; i < H * H / TB; ++i) v[i] = __bfloat162float(W[OFF_W2 + threadIdx.x + i * TB]);
#pragma unroll
        for (int i = 0; i < H * H / TB; ++i) sW2[threadIdx.x + i * TB] = v[i];                   // [out][in]
    }
    const int tx = fast_side(), ty = slow_side(), c0 = ty * 4, r0 = tx * 4;
    const auto relu = [](float v, int, int) { return fmaxf(v, 0.f); };
    f2 g2[4][4] = {}, g1[4] = {};                                 // sums of the even rows and of the odd ones
    float gs = 0.f, g3 = 0.f;
    const long long b = blockIdx.x, part = tiles / gridDim.x, more = tiles % gridDim.x;
    const long long begin = (b * part + min(b, more)) * TR, end = min(n, begin + (part + (b < more ? 1 : 0)) * TR);
    const bool wide = (reinterpret_cast<uintptr_t>(X) & 15u) == 0;
    const int dr = threadIdx.x / O, dc = threadIdx.x % O;         // sO [output][row]; zeros past the end
    auto load_d = [&](long long row) { return threadIdx.x < TR * O && row + dr < end ? dOut[(row + dr) * O + dc] : 0.f; };
    float4 xn = load_rows(end, begin, X, wide);
    float dn = load_d(begin);
    // The rows past the end have activations too (the biases'); they are no one's rows, and zeros would
    // not keep an infinite one out of the sums.  A thread clears the entries that it stored.
    auto clear_past = [&](float *out, long long left) {
        if (left >= TR) return;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (r0 + i >= left)
#pragma unroll
                for (int j = 0; j < 4; ++j) out[(c0 + j) * LD + r0 + i] = 0.f;
    };
    for (long long row = begin; row < end; row += TR) {
        __syncthreads();
        stage_rows(xn, sX);
        if (threadIdx.x < TR * O) sO[dc * TR + dr] = dn;
        xn = load_rows(end, row + TR, X, wide);
        dn = load_d(row + TR);
        __syncthreads();
        float acc[4][4];
        tile_gemm<F>(sX, sW + SW1, sW + SB1, r0, c0, acc);
        tile_store(sH1, r0, c0, acc, relu);
        clear_past(sH1, end - row);
        __syncthreads();
        tile_gemm<H>(sH1, sW + SW2, sW + SB2, r0, c0, acc);
        tile_store(sH2, r0, c0, acc, relu);
        tile_store(sD2, r0, c0, acc, [&](float z, int i, int j) {
            const float dh = fmaf(sW[SW3 + c0 + j], sO[r0 + i], sW[SW3 + H + c0 + j] * sO[TR + r0 + i]);
            return z > 0.f ? dh : 0.f;
        });
        clear_past(sH2, end - row);
        clear_past(sD2, end - row);
        __syncthreads();
        tile_gemm<H>(sD2, sW2, nullptr, r0, c0, acc);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 h = *reinterpret_cast<const float4 *>(sH1 + (c0 + j) * LD + r0);
            *reinterpret_cast<float4 *>(sD1 + (c0 + j) * LD + r0) =
                make_float4(h.x > 0.f ? acc[0][j] : 0.f, h.y > 0.f ? acc[1][j] : 0.f, h.z > 0.f ? acc[2][j] : 0.f, h.w > 0.f ? acc[3][j] : 0.f);
        }
        __syncthreads();
#pragma unroll 2
        for (int r = 0; r < TR; r += 4) {
            ulonglong2 d2[4], h1[4], d1[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                d2[i] = *reinterpret_cast<const ulonglong2 *>(sD2 + (ty + 16 * i) * LD + r);
                h1[i] = *reinterpret_cast<const ulonglong2 *>(sH1 + (tx + 16 * i) * LD + r);
                d1[i] = *reinterpret_cast<const ulonglong2 *>(sD1 + (ty + 16 * i) * LD + r);
            }
            const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(sX + tx * LD + r);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    g2[i][j] = fma2(d2[i].x, h1[j].x, g2[i][j]);
                    g2[i][j] = fma2(d2[i].y, h1[j].y, g2[i][j]);
                }
                g1[i] = fma2(d1[i].x, x.x, g1[i]);
                g1[i] = fma2(d1[i].y, x.y, g1[i]);
            }
        }
        {
            const int k = threadIdx.x;
            const float *src = (k < H ? sD1 + k * LD : k < 2 * H ? sD2 + (k - H) * LD : sH2 + (k % H) * LD);
            const float *d = sO + (k < 3 * H ? 0 : TR);
#pragma unroll 4
            for (int r = 0; r < TR; r += 4) {
                const float4 v = *reinterpret_cast<const float4 *>(src + r);
                if (k < 2 * H) {
                    gs += v.x; gs += v.y; gs += v.z; gs += v.w;
                } else {
                    gs = fmaf(d[r], v.x, gs); gs = fmaf(d[r + 1], v.y, gs);
                    gs = fmaf(d[r + 2], v.z, gs); gs = fmaf(d[r + 3], v.w, gs);
                }
            }
            if (k < TR) g3 += sO[(k >> 5) * TR + (k & 31)] + sO[(k >> 5) * TR + (k & 31) + 32];   // warp o: output o
        }
    }
    float *out = partials + static_cast<long long>(blockIdx.x) * NPARAM;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float2 v = unpack(g2[i][j]);
            out[OFF_W2 + (ty + 16 * i) * H + tx + 16 * j] = v.x + v.y;
        }
        const float2 v = unpack(g1[i]);
        out[OFF_W1 + (ty + 16 * i) * F + tx] = v.x + v.y;
    }
    const int k = threadIdx.x;
    out[k < H ? OFF_B1 + k : k < 2 * H ? OFF_B2 + k - H : OFF_W3 + k - 2 * H] = gs;
    if (k < TR) {
        for (int w = 16; w > 0; w >>= 1) g3 += __shfl_down_sync(0xFFFFFFFFu, g3, w);
        if ((k & 31) == 0) out[OFF_B3 + (k >> 5)] = g3;
    }
}

// grad[k] = the sum of the chunks' partials: 8 threads per parameter take every eighth chunk, then
// their sums in order.
__global__ void mlp_reduce_partials_kernel(int chunks, const float *partials, float *grad) {
    __shared__ float part[8][32];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, k = blockIdx.x * 32 + lane;
    float acc = 0.f;
    if (k < NPARAM) {
#pragma unroll 8
        for (int c = g; c < chunks; c += 8) acc += partials[static_cast<long long>(c) * NPARAM + k];
    }
    part[g][lane] = acc;
    __syncthreads();
    if (g == 0 && k < NPARAM) {
        acc = part[0][lane];
#pragma unroll
        for (int i = 1; i < 8; ++i) acc += part[i][lane];
        grad[k] = acc;
    }
}

// Loss per segment (instance) and dOut: cross-entropy of softmax(o_1) to target_w plus the mean
// binary cross-entropy of sigmoid(o_2) to target_p, each segment weighted 1 / n_seg.
__global__ void mlp_loss_kernel(int n_seg, const long long *seg, const float *Out,
                                const float *target_w, const float *target_p, float *dOut,
                                double *loss_seg) {
    const int s = blockIdx.x;
    const long long a = seg[s], b = seg[s + 1];
    __shared__ float red[256];
    __shared__ double redd[256];
    float mx = -3.0e38f;
    for (long long r = a + threadIdx.x; r < b; r += blockDim.x) mx = fmaxf(mx, Out[r * O]);
    red[threadIdx.x] = mx;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] = fmaxf(red[threadIdx.x], red[threadIdx.x + w]);
        __syncthreads();
    }
    mx = red[0];
    __syncthreads();
    float se = 0.f, st = 0.f;
    for (long long r = a + threadIdx.x; r < b; r += blockDim.x) { se += __expf(Out[r * O] - mx); st += target_w[r]; }
    red[threadIdx.x] = se;
    redd[threadIdx.x] = st;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) { red[threadIdx.x] += red[threadIdx.x + w]; redd[threadIdx.x] += redd[threadIdx.x + w]; }
        __syncthreads();
    }
    const float lse = mx + __logf(red[0]);
    const float tsum = static_cast<float>(redd[0]);
    __syncthreads();
    const float inv_seg = 1.f / n_seg, inv_len = 1.f / static_cast<float>(b - a);
    double part = 0.0;
    for (long long r = a + threadIdx.x; r < b; r += blockDim.x) {
        const float o1 = Out[r * O], z = Out[r * O + 1], t = target_w[r], p = target_p[r];
        const float sm = __expf(o1 - lse);
        dOut[r * O] = (sm * tsum - t) * inv_seg;
        const float sig = 1.f / (1.f + __expf(-z));
        dOut[r * O + 1] = (sig - p) * inv_len * inv_seg;
        const float softplus = z > 0.f ? z + log1pf(__expf(-z)) : log1pf(__expf(z));
        part += static_cast<double>(-t * (o1 - lse)) + static_cast<double>((softplus - p * z) * inv_len);
    }
    redd[threadIdx.x] = part;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) redd[threadIdx.x] += redd[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) loss_seg[s] = redd[0] / n_seg;
}

__global__ void mlp_adam_kernel(int step, float lr, float b1, float b2, float eps, float *master,
                                float *m, float *v, const float *grad, __nv_bfloat16 *W) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= NPARAM) return;
    const float g = grad[k];
    const float mk = b1 * m[k] + (1.f - b1) * g;
    const float vk = b2 * v[k] + (1.f - b2) * g * g;
    m[k] = mk;
    v[k] = vk;
    const float mhat = mk / (1.f - powf(b1, static_cast<float>(step)));
    const float vhat = vk / (1.f - powf(b2, static_cast<float>(step)));
    master[k] -= lr * mhat / (sqrtf(vhat) + eps);
    W[k] = __float2bfloat16_rn(master[k]);
}

__global__ void mlp_cast_kernel(const float *master, __nv_bfloat16 *W) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < NPARAM) W[k] = __float2bfloat16_rn(master[k]);
}

// Heads per segment: w = 0.5 softmax(o_1) + 0.5 / n, nu = clamp(sigmoid(o_2)).
__global__ void mlp_heads_kernel(const long long *seg, const float *Out, double *w, double *nu) {
    const int s = blockIdx.x;
    const long long a = seg[s], b = seg[s + 1];
    __shared__ double red[256];
    double mx = -1e300;
    for (long long r = a + threadIdx.x; r < b; r += blockDim.x) mx = fmax(mx, static_cast<double>(Out[r * O]));
    red[threadIdx.x] = mx;
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if (threadIdx.x < k) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + k]);
        __syncthreads();
    }
    mx = red[0];
    __syncthreads();
    double se = 0.0;
    for (long long r = a + threadIdx.x; r < b; r += blockDim.x) se += exp(static_cast<double>(Out[r * O]) - mx);
    red[threadIdx.x] = se;
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    const double tot = red[0];
    const double n = static_cast<double>(b - a);
    for (long long r = a + threadIdx.x; r < b; r += blockDim.x) {
        w[r] = 0.5 * (exp(static_cast<double>(Out[r * O]) - mx) / tot) + 0.5 / n;
        const double sg = 1.0 / (1.0 + exp(-static_cast<double>(Out[r * O + 1])));
        nu[r] = fmin(fmax(sg, 1e-6), 1.0 - 1e-6);
    }
}

// Features.  The designs lie one after the other as the caller holds them: instance s's clone_ptr at
// ptr + clone_off[s] + s (local offsets), its entries from pools + entry_off[s], its pools from
// pool_off[s] on.
struct FeatIn {
    const int32_t *ptr, *pools;
    const uint8_t *y;
    const long long *clone_off, *entry_off, *pool_off;   // [n_inst + 1]
    const double *consts;                                 // [n_inst][4]: lambda, a+, a-, mean pool size
    int n_inst;
    int32_t *psize, *ap_pool, *nap;                       // pool sizes, all-positive clones per pool and per instance
};
struct FeatClone { int s; const int32_t *row; int d; long long base; };
// Clone i: its instance (binary search), its pools, the first pool of its instance.
__device__ __forceinline__ FeatClone feat_clone(const FeatIn &in, long long i) {
    int lo = 0, hi = in.n_inst - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (in.clone_off[mid] <= i) lo = mid; else hi = mid - 1;
    }
    const int32_t *p = in.ptr + i + lo;
    const int32_t e0 = p[0] - in.ptr[in.clone_off[lo] + lo];
    return {lo, in.pools + in.entry_off[lo] + e0, p[1] - p[0], in.pool_off[lo]};
}
__device__ __forceinline__ int feat_positive(const FeatIn &in, const FeatClone &c) {
    int p = 0;
    for (int e = 0; e < c.d; ++e) p += in.y[c.base + c.row[e]] ? 1 : 0;
    return p;
}

// Pool sizes; per pool and per instance the clones all of whose pools are positive.
__global__ void feat_counts(long long n, const FeatIn in) {
    const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const FeatClone c = feat_clone(in, i);
    const bool all = c.d > 0 && feat_positive(in, c) == c.d;
    for (int e = 0; e < c.d; ++e) {
        atomicAdd(&in.psize[c.base + c.row[e]], 1);
        if (all) atomicAdd(&in.ap_pool[c.base + c.row[e]], 1);
    }
    if (all) atomicAdd(&in.nap[c.s], 1);
}

__global__ void feat_rows(long long n, const FeatIn in, float *Fout) {
    const long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const FeatClone c = feat_clone(in, i);
    const double lam = in.consts[4 * c.s], a_pos = in.consts[4 * c.s + 1], a_neg = in.consts[4 * c.s + 2], dbar = in.consts[4 * c.s + 3];
    const int d = c.d, p = feat_positive(in, c), nn = d - p, ap = d > 0 && p == d ? 1 : 0;
    double sum_d = 0.0, sum_dpos = 0.0, sum_inv = 0.0;
    int min_ap = 1 << 30, sole = 0, unexplained = 0;
    for (int e = 0; e < d; ++e) {
        const long long j = c.base + c.row[e];
        const int size = in.psize[j];
        sum_d += size;
        if (in.y[j]) {
            const int a = in.ap_pool[j];
            sum_dpos += size;
            min_ap = min(min_ap, a);
            sum_inv += 1.0 / max(a, 1);
            if (ap && a == 1) ++sole;
            if (a == 0) ++unexplained;
        }
    }
    const float4 f[4] = {
        make_float4(d / 8.0f, p / 8.0f, nn / 8.0f, static_cast<float>(p) / static_cast<float>(max(d, 1))),
        make_float4(static_cast<float>((lam + p * a_pos + nn * a_neg) / 10.0), d ? static_cast<float>(sum_d / d / dbar) : 0.f,
                    p ? static_cast<float>(sum_dpos / p / dbar) : 0.f, static_cast<float>(ap)),
        make_float4(p ? min_ap / 10.0f : 0.f, p ? static_cast<float>(sum_inv / p) : 0.f, sole / 8.0f, unexplained / 8.0f),
        make_float4(in.nap[c.s] / 100.0f, static_cast<float>(lam / 10.0), static_cast<float>(a_pos / 10.0),
                    static_cast<float>(a_neg / 10.0))};
    float *out = Fout + i * 16;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if ((reinterpret_cast<uintptr_t>(Fout) & 15u) == 0) {
            reinterpret_cast<float4 *>(out)[k] = f[k];
        } else {                       // the caller's array need only hold floats
            out[4 * k] = f[k].x; out[4 * k + 1] = f[k].y; out[4 * k + 2] = f[k].z; out[4 * k + 3] = f[k].w;
        }
    }
}

int grid_for(long long n, int block) {
    long long g = (n + block - 1) / block;
    return static_cast<int>(g < 1 ? 1 : (g > 65535LL * 64 ? 65535LL * 64 : g));
}

}  // namespace
}  // namespace mcpd

namespace {
int fail_m(mcpd_ctx *ctx, int code, const std::string &msg) {
    if (ctx) ctx->err = msg;
    return code;
}
}  // namespace

#define CUM(call)                                                                                 \
    do {                                                                                          \
        cudaError_t e_ = (call);                                                                  \
        if (e_ != cudaSuccess) return fail_m(ctx, MCPD_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

extern "C" {

int mcpd_mlp_num_params(void) { return mcpd::NPARAM; }

int mcpd_features_batch(mcpd_ctx *ctx, int32_t n_inst, const mcpd_design *designs,
                        const uint8_t *const *ys, const double *rates, float *feat_dev) {
    using namespace mcpd;
    if (!ctx || n_inst < 1 || !designs || !ys || !rates || !feat_dev) return MCPD_EINVAL;
    // Sizes and checks.
    std::vector<long long> off(3 * (static_cast<size_t>(n_inst) + 1), 0);
    long long *const clone_off = off.data(), *const entry_off = clone_off + n_inst + 1, *const pool_off = entry_off + n_inst + 1;
    std::vector<double> consts(4 * static_cast<size_t>(n_inst));
    for (int32_t s = 0; s < n_inst; ++s) {
        const mcpd_design &d = designs[s];
        if (d.n_clones < 1 || d.n_pools < 1 || !d.clone_ptr) return fail_m(ctx, MCPD_EINVAL, "bad design");
        const double fp = rates[3 * s], fn = rates[3 * s + 1], q = rates[3 * s + 2];
        if (!(fp > 0 && fp < 1 && fn > 0 && fn < 1 && q > 0 && q < 1)) return fail_m(ctx, MCPD_EINVAL, "rates out of (0,1)");
        consts[4 * s] = std::log(q) - std::log(1.0 - q);
        consts[4 * s + 1] = std::log(1.0 - fn) - std::log(fp);
        consts[4 * s + 2] = std::log(fn) - std::log(1.0 - fp);
        consts[4 * s + 3] = static_cast<double>(d.clone_ptr[d.n_clones]) / d.n_pools;
        long long entries = 0;
        for (int32_t i = 0; i < d.n_clones; ++i) entries += std::max(0, d.clone_ptr[i + 1] - d.clone_ptr[i]);
        clone_off[s + 1] = clone_off[s] + d.n_clones;
        entry_off[s + 1] = entry_off[s] + entries;
        pool_off[s + 1] = pool_off[s] + d.n_pools;
    }
    const long long n = clone_off[n_inst], entries = entry_off[n_inst], pools = pool_off[n_inst];
    // One upload: offsets, constants, clone_ptr and clone_pools as they are, outcomes; then the device's
    // counts.  (Pool bases and instances written per clone on the host, six pageable copies and an
    // allocation per call took 1.5 ms for 64 instances of 1298 clones.)
    size_t bytes = 0;
    auto take = [&](size_t b) { const size_t at = bytes; bytes += (b + 15) / 16 * 16; return at; };
    const size_t o_off = take(off.size() * 8), o_consts = take(consts.size() * 8), o_ptr = take((n + n_inst) * 4);
    const size_t o_pools = take(entries * 4), o_y = take(pools), uploaded = bytes;
    const size_t o_count = take((2 * pools + n_inst) * 4);
    CUM(cudaSetDevice(ctx->device));
    if (bytes > ctx->stage_bytes) {
        if (ctx->stage_bytes) { cudaFreeHost(ctx->stage_host); cudaFree(ctx->stage_dev); ctx->stage_bytes = 0; }
        CUM(cudaMallocHost(&ctx->stage_host, bytes));
        const cudaError_t e = cudaMalloc(&ctx->stage_dev, bytes);
        if (e != cudaSuccess) { cudaFreeHost(ctx->stage_host); return fail_m(ctx, MCPD_ECUDA, "cudaMalloc"); }
        ctx->stage_bytes = bytes;
    }
    char *const h = static_cast<char *>(ctx->stage_host), *const dv = static_cast<char *>(ctx->stage_dev);
    std::memcpy(h + o_off, off.data(), off.size() * 8);
    std::memcpy(h + o_consts, consts.data(), consts.size() * 8);
    int rc = MCPD_OK;
    for (int32_t s = 0; s < n_inst && rc == MCPD_OK; ++s) {
        const mcpd_design &d = designs[s];
        int32_t *ptr = reinterpret_cast<int32_t *>(h + o_ptr) + clone_off[s] + s;
        int32_t *pl = reinterpret_cast<int32_t *>(h + o_pools) + entry_off[s];
        uint32_t worst = 0;
        if (entry_off[s + 1] - entry_off[s] == d.clone_ptr[d.n_clones] - d.clone_ptr[0]) {      // ascending
            std::memcpy(ptr, d.clone_ptr, (static_cast<size_t>(d.n_clones) + 1) * 4);
            const int32_t *src = d.clone_pools + d.clone_ptr[0];
            for (long long e = 0, m = entry_off[s + 1] - entry_off[s]; e < m; ++e) {
                worst = std::max(worst, static_cast<uint32_t>(src[e]));
                pl[e] = src[e];
            }
        } else {                       // a falling clone_ptr: the clone has no pools
            int32_t at = 0;
            for (int32_t i = 0; i < d.n_clones; ++i) {
                ptr[i] = at;
                for (int32_t e = d.clone_ptr[i]; e < d.clone_ptr[i + 1]; ++e) {
                    worst = std::max(worst, static_cast<uint32_t>(d.clone_pools[e]));
                    pl[at++] = d.clone_pools[e];
                }
            }
            ptr[d.n_clones] = at;
        }
        if (entry_off[s + 1] > entry_off[s] && worst >= static_cast<uint32_t>(d.n_pools)) rc = fail_m(ctx, MCPD_EINVAL, "pool id");
        std::memcpy(h + o_y + pool_off[s], ys[s], static_cast<size_t>(d.n_pools));
    }
    if (rc == MCPD_OK) {
        cudaStream_t st = ctx->stream;
        FeatIn in;
        in.clone_off = reinterpret_cast<const long long *>(dv + o_off);
        in.entry_off = in.clone_off + n_inst + 1;
        in.pool_off = in.entry_off + n_inst + 1;
        in.consts = reinterpret_cast<const double *>(dv + o_consts);
        in.ptr = reinterpret_cast<const int32_t *>(dv + o_ptr);
        in.pools = reinterpret_cast<const int32_t *>(dv + o_pools);
        in.y = reinterpret_cast<const uint8_t *>(dv + o_y);
        in.n_inst = n_inst;
        in.psize = reinterpret_cast<int32_t *>(dv + o_count);
        in.ap_pool = in.psize + pools;
        in.nap = in.ap_pool + pools;
        const int g = grid_for(n, 256);
        if (cudaMemcpyAsync(dv, h, uploaded, cudaMemcpyHostToDevice, st) != cudaSuccess ||
            cudaMemsetAsync(in.psize, 0, (2 * pools + n_inst) * 4, st) != cudaSuccess) {
            rc = MCPD_ECUDA;
        } else {
            feat_counts<<<g, 256, 0, st>>>(n, in);
            feat_rows<<<g, 256, 0, st>>>(n, in, feat_dev);
            if (cudaGetLastError() != cudaSuccess) rc = MCPD_ECUDA;
        }
        if (cudaStreamSynchronize(st) != cudaSuccess) rc = MCPD_ECUDA;
        if (rc != MCPD_OK) fail_m(ctx, rc, "features kernels");
    }
    if (ctx->stage_bytes > kKeepStaging) {
        cudaFreeHost(ctx->stage_host);
        cudaFree(ctx->stage_dev);
        ctx->stage_host = ctx->stage_dev = nullptr;
        ctx->stage_bytes = 0;
    }
    return rc;
}

int mcpd_mlp_forward(mcpd_ctx *ctx, int64_t n_rows, const float *X, const uint16_t *W, float *Out) {
    using namespace mcpd;
    if (!ctx || n_rows < 0 || (n_rows && (!X || !W || !Out))) return MCPD_EINVAL;
    CUM(cudaSetDevice(ctx->device));
    if (n_rows == 0) return MCPD_OK;
    CUM(cudaFuncSetAttribute(mlp_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FWD_SMEM));
    const int g = static_cast<int>(std::min<long long>((n_rows + TR - 1) / TR, 3LL * ctx->sm_count));
    mlp_forward_kernel<<<g, TB, FWD_SMEM, ctx->stream>>>(n_rows, X, reinterpret_cast<const __nv_bfloat16 *>(W), Out);
    CUM(cudaGetLastError());
    return MCPD_OK;
}

int mcpd_mlp_loss(mcpd_ctx *ctx, int32_t n_seg, const int64_t *seg_dev, const float *Out,
                  const float *target_w, const float *target_p, float *dOut, double *loss_seg_dev) {
    if (!ctx || n_seg < 1 || !seg_dev || !Out || !target_w || !target_p || !dOut || !loss_seg_dev) return MCPD_EINVAL;
    CUM(cudaSetDevice(ctx->device));
    mcpd::mlp_loss_kernel<<<n_seg, 256, 0, ctx->stream>>>(n_seg, reinterpret_cast<const long long *>(seg_dev), Out,
                                                           target_w, target_p, dOut, loss_seg_dev);
    CUM(cudaGetLastError());
    return MCPD_OK;
}

int mcpd_mlp_backward(mcpd_ctx *ctx, int64_t n_rows, const float *X, const uint16_t *W,
                      const float *dOut, float *work, int64_t work_floats, float *grad) {
    using namespace mcpd;
    if (!ctx || n_rows < 1 || !X || !W || !dOut || !work || !grad) return MCPD_EINVAL;
    const long long chunks = chunks_of(n_rows);
    if (work_floats < chunks * NPARAM) return fail_m(ctx, MCPD_EINVAL, "backward workspace too small");
    CUM(cudaSetDevice(ctx->device));
    CUM(cudaFuncSetAttribute(mlp_backward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BWD_SMEM));
    mlp_backward_kernel<<<static_cast<unsigned>(chunks), TB, BWD_SMEM, ctx->stream>>>(
        n_rows, tiles_of(n_rows), X, reinterpret_cast<const __nv_bfloat16 *>(W), dOut, work);
    mlp_reduce_partials_kernel<<<(NPARAM + 31) / 32, 256, 0, ctx->stream>>>(static_cast<int>(chunks), work, grad);
    CUM(cudaGetLastError());
    return MCPD_OK;
}

int64_t mcpd_mlp_backward_workspace(int64_t n_rows) {
    if (n_rows < 1) return 0;
    return mcpd::chunks_of(n_rows) * mcpd::NPARAM;
}

int mcpd_mlp_adam(mcpd_ctx *ctx, int32_t step, float lr, float beta1, float beta2, float eps,
                  float *master, float *m, float *v, const float *grad, uint16_t *W) {
    if (!ctx || step < 1 || !master || !m || !v || !grad || !W) return MCPD_EINVAL;
    CUM(cudaSetDevice(ctx->device));
    mcpd::mlp_adam_kernel<<<(mcpd::NPARAM + 255) / 256, 256, 0, ctx->stream>>>(
        step, lr, beta1, beta2, eps, master, m, v, grad, reinterpret_cast<__nv_bfloat16 *>(W));
    CUM(cudaGetLastError());
    return MCPD_OK;
}

int mcpd_mlp_cast(mcpd_ctx *ctx, const float *master, uint16_t *W) {
    if (!ctx || !master || !W) return MCPD_EINVAL;
    CUM(cudaSetDevice(ctx->device));
    mcpd::mlp_cast_kernel<<<(mcpd::NPARAM + 255) / 256, 256, 0, ctx->stream>>>(master, reinterpret_cast<__nv_bfloat16 *>(W));
    CUM(cudaGetLastError());
    return MCPD_OK;
}

int mcpd_mlp_heads(mcpd_ctx *ctx, int32_t n_seg, const int64_t *seg_dev, const float *Out,
                   double *w_dev, double *nu_dev) {
    if (!ctx || n_seg < 1 || !seg_dev || !Out || !w_dev || !nu_dev) return MCPD_EINVAL;
    CUM(cudaSetDevice(ctx->device));
    mcpd::mlp_heads_kernel<<<n_seg, 256, 0, ctx->stream>>>(reinterpret_cast<const long long *>(seg_dev), Out, w_dev, nu_dev);
    CUM(cudaGetLastError());
    return MCPD_OK;
}

}  // extern "C"
