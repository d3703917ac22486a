// Stand-alone GEMM for a few rows on the caller's own row-major operands: Y[M][N] = X[M][K] * W[N][K]^T, M <= 32.
#pragma once
#include "ptx.cuh"

namespace sdv {

constexpr int kSmallGemmWarps = 8;

// A cluster takes 16 rows of W; its blocks' warps take the 32-column steps of K in turn (step t goes to warp t mod all warps)
// and read both operands straight into registers: the order of the products inside a step is free, so every lane loads
// eight consecutive values per row and uses them as the fragments of two m16n8k16 instructions (the weights are the 16
// rows, NT tiles of 8 token rows the columns; X is rounded to bf16 on the way).  The warps' sums meet in shared memory,
// the blocks' through distributed shared memory: no scratch in global memory, nothing to clear, one launch.
// Bound by its latency: launch, one round trip to memory, two block barriers (4 us on the device at 9 x 640 x 768; with a
// packing pass, two clears and a copy around the weight-streaming kernel a call took 56 us).
template <int NT>
__global__ void __launch_bounds__(kSmallGemmWarps * 32) small_gemm_kernel(const float* x, const uint16_t* w, float* y, int M, int N, int K) {
    constexpr int LD = NT * 8 + 1;
    __shared__ float part[kSmallGemmWarps][16][LD];
    __shared__ float sum[16][LD];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const int CS = (int)cluster_size(), rank = (int)cluster_rank();
    const int n0 = ((int)blockIdx.x / CS) * 16, steps = K / 32, stride = CS * kSmallGemmWarps;
    const uint16_t* w0 = w + (size_t)(n0 + g) * K + q * 8;
    const uint16_t* w1 = w0 + (size_t)8 * K;
    const float* xr[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) xr[t] = x + (size_t)min(t * 8 + g, M - 1) * K + q * 8;   // rows past M repeat the last, not used
    float d[NT][4];
#pragma unroll
    for (int t = 0; t < NT; ++t) d[t][0] = d[t][1] = d[t][2] = d[t][3] = 0.f;
    constexpr int U = NT <= 2 ? 4 : 2;   // steps whose loads are in flight together
    for (int s0 = rank * kSmallGemmWarps + warp; s0 < steps; s0 += U * stride) {
        uint4 a0[U], a1[U];
        float4 b0[U][NT], b1[U][NT];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int s = s0 + u * stride;
            if (s < steps) {
                a0[u] = __ldg(reinterpret_cast<const uint4*>(w0 + s * 32));
                a1[u] = __ldg(reinterpret_cast<const uint4*>(w1 + s * 32));
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    b0[u][t] = __ldg(reinterpret_cast<const float4*>(xr[t] + s * 32));
                    b1[u][t] = __ldg(reinterpret_cast<const float4*>(xr[t] + s * 32 + 4));
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (s0 + u * stride < steps) {
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                    const uint32_t p0 = pack_bf16(b0[u][t].x, b0[u][t].y), p1 = pack_bf16(b0[u][t].z, b0[u][t].w);
                    const uint32_t p2 = pack_bf16(b1[u][t].x, b1[u][t].y), p3 = pack_bf16(b1[u][t].z, b1[u][t].w);
                    mma_bf16_16816(d[t], a0[u].x, a1[u].x, a0[u].y, a1[u].y, p0, p1);
                    mma_bf16_16816(d[t], a0[u].z, a1[u].z, a0[u].w, a1[u].w, p2, p3);
                }
            }
        }
    }
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        part[warp][g][t * 8 + q * 2] = d[t][0];
        part[warp][g][t * 8 + q * 2 + 1] = d[t][1];
        part[warp][g + 8][t * 8 + q * 2] = d[t][2];
        part[warp][g + 8][t * 8 + q * 2 + 1] = d[t][3];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 16 * M; i += kSmallGemmWarps * 32) {
        const int n = i & 15, m = i >> 4;
        float v = 0.f;
#pragma unroll
        for (int k = 0; k < kSmallGemmWarps; ++k) v += part[k][n][m];
        if (CS == 1) y[(size_t)m * N + n0 + n] = v;
        else sum[n][m] = v;
    }
    if (CS > 1) {
        cluster_sync();
        for (int i = rank * kSmallGemmWarps * 32 + threadIdx.x; i < 16 * M; i += stride * 32) {
            const int n = i & 15, m = i >> 4;
            float v = 0.f;
            for (int k = 0; k < CS; ++k) v += ld_cluster_f1(map_shared_rank(smem_u32(&sum[n][m]), k));
            y[(size_t)m * N + n0 + n] = v;
        }
        __syncwarp();
        cluster_sync();   // no block leaves while another still reads its sums
    }
}

}  // namespace sdv
