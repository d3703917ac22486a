// Dense prefill path: a sub-chunk of the request (up to 1024 tokens) through the decoder as plain matrix
// products on the tensor cores.  The verify kernel puts the few token rows on the N side of the
// instruction and streams every weight once per launch; a prefill chunk has enough rows to fill the M
// side instead.  A layer is eight kernels, each launched while the one before it still runs
// (programmatic dependent launch: a kernel sets itself up, products even fetch their first weight tiles,
// and then waits for its inputs):
//     q|k|v product -> K-share sums, bias, rotary embedding, KV append -> attention -> output projection ->
//     K-share sums, residual, norm -> gate|up product with SwiGLU -> down projection -> sums, residual, norm
// The products (dense_gemm_kernel) run on pairs of SMs; products with few output tiles split K and leave
// fp32 partial sums that the next, row-wise kernel adds up while it reads them anyway.
#pragma once
#include <cuda.h>
#include <math_constants.h>

#include "layout.cuh"
#include "ptx.cuh"

namespace sdv {

constexpr int kDenseBK = 64;            // input features per stage: 64 bf16 = one 128-byte swizzled row
constexpr int kDenseMaxRows = 1024;     // rows of the activation buffers (one sub-chunk)
constexpr int kDenseMaxSplits = 16;     // K shares of one product at most
constexpr int kDenseTopMax = 4;         // best logits kept per row and vocabulary tile (calibration)

enum DenseEpilogue { EPI_PARTIAL = 0, EPI_SWIGLU = 1, EPI_TOP = 2 };
// Warp 0: copies, warp 1: tensor-core issue, the others: epilogue, two warps per 32 rows where a value takes more than its
// store (best logits of 256 rows x 151936 ids: 105 -> 69 us, SwiGLU 16.0 -> 15.8 us; plain partial sums 8.4 -> 8.6, so one there)
template <int EPI>
constexpr int kDenseHalves = EPI == EPI_PARTIAL ? 1 : 2;
template <int EPI>
constexpr int kDenseThreads = 64 + 128 * kDenseHalves<EPI>;

constexpr int kDenseTurnLd = 36;                                // floats; an odd number of 16-byte units spreads the rows over the banks
constexpr int kDenseTurnBytes = 32 * kDenseTurnLd * 4;          // 32 rows x 32 columns of partial sums on their way out, per warp

// Stage of a pair tile of 256 tokens x BN features: every SM of the pair holds 128 token rows and half of the
// features' weight rows.
template <int BN>
struct DenseShape {
    static constexpr int kABytes = 128 * kDenseBK * 2;
    static constexpr int kBBytes = BN / 2 * kDenseBK * 2;
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kStages = BN == 256 ? 6 : 8;
    static constexpr int kSmemBytes = kStages * kStageBytes + 1024 + 512 + (BN == 128 ? 4 * kDenseTurnBytes : 0);
};

struct DenseTopOut {   // EPI_TOP: [row][share of the vocabulary: pair, part of its columns][kDenseTopMax] best logits of the share and their ids, best first
    float* val;
    int* idx;
};

// C[m][n] = sum_k A[m][k] * B[n][k]; A = activations (bf16, row-major [rows][K]), B = weights (bf16, row-major
// [N][K]).  One cluster of two SMs works on a 256 (tokens) x BN (features) tile with cta_group::2
// instructions: each SM copies its 128 token rows and half of the weight rows per 64-column stage, the leading
// SM's thread issues, and each SM ends up with its 128 rows x BN accumulator in its own tensor memory (two
// buffers, so the next tile's products run while this one is read out).  Against one 128 x 128 tile per SM this
// halves the bytes every SM pulls from L2 per flop and the shared-memory reads per instruction.
// Pairs walk the tiles persistently: (features, 256-row tokens, K share), K shares fastest.
//   EPI_PARTIAL: part[z][m][n] = the share's sum (row stride N)
//   EPI_SWIGLU:  features come as 64 gate rows then the 64 matching up rows: out_bf16[m][64 t + c] = silu(gate) * up
//   EPI_TOP:     the best kDenseTopMax values of every row over the tiles this pair walks (largest first, lowest id first
//                among equals): a pair stays with its 256 rows, so a thread keeps its row's best in registers and most
//                values only take part in a maximum over 32
// Rows >= M and columns >= N are computed on whatever the copies deliver (zeros outside the tensors) and
// never written.  err: set to 1 when a bounded wait runs out.
// Measured on B200 (BN 256, 1536 x 17920 weights): 256 tokens 18.6 us stand-alone (758 TFLOP/s; 25.4 us with
// 128 x 128 tiles on single SMs), 1024 tokens 41 us (1371 TFLOP/s).  With 256 tokens the weights' HBM read
// (8.4 us) and the fill and drain of the pipeline bound it, with 1024 the tensor cores.
template <int EPI, int BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kDenseThreads<EPI>, 1)
dense_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, int M, int N, int K,
                  int splits, float* part, __nv_bfloat16* out_bf16, int ld_bf16, DenseTopOut top, int* err,
                  unsigned long long wait_limit_ns) {
    using S = DenseShape<BN>;
    constexpr int kHalves = kDenseHalves<EPI>;
    extern __shared__ uint8_t dense_smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dense_smem_raw) + 1023) & ~(uintptr_t)1023);
    struct Ctl {
        uint64_t full[S::kStages], empty[S::kStages];  // full: the leading SM's counts both SMs' bytes
        uint64_t acc_full[2], acc_empty[2];            // acc_empty: the leading SM's counts both SMs' epilogue warps
        uint64_t stopped;                              // behind an abandoned wait: the products issued before it have completed
        uint32_t tmem_base;
        int abort_flag;
    };
    Ctl* ctl = reinterpret_cast<Ctl*>(smem + S::kStages * S::kStageBytes);
    static_assert(sizeof(Ctl) <= 512, "control block");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int mt = (M + 255) / 256, nt = (N + BN - 1) / BN, ntiles = mt * nt * splits;
    const int nkb_all = K / kDenseBK;
    const int pair = (int)blockIdx.x >> 1;
    int npairs = (int)gridDim.x >> 1;   // stride of the walk
    if (EPI == EPI_TOP) npairs = npairs / mt * mt;
    const int t0 = pair < npairs ? pair : ntiles;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S::kStages; ++s) {
            mbar_init(&ctl->full[s], 1);
            mbar_init(&ctl->empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&ctl->acc_full[b], 1);
            mbar_init(&ctl->acc_empty[b], 8 * kHalves);
        }
        mbar_init(&ctl->stopped, 1);
        ctl->abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 1) tmem_alloc_pair(&ctl->tmem_base, 512);
    tc_fence_before();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    grid_dep_launch();

    if (warp == 0) {
        if (elect_one()) {
            uint32_t s = 0, par = 0, issued = 0;
            bool ok = true, first = true;
            for (int t = t0; t < ntiles && ok; t += npairs) {
                const int z = t % splits, r = t / splits;
                const int m0 = (r % mt) * 256 + (int)rank * 128, n0 = (r / mt) * BN + (int)rank * (BN / 2);
                const int kb0 = even_start(nkb_all, splits, z), nkb = even_count(nkb_all, splits, z);
                int kb = 0;
                if (first) {
                    // the weights do not depend on the kernel before: the first ring's worth is fetched while it still runs
                    first = false;
                    const int n1 = nkb < S::kStages ? nkb : S::kStages;
                    for (int i = 0; i < n1; ++i) {
                        if (rank == 0) mbar_arrive_expect_tx(&ctl->full[i], 2 * S::kStageBytes);
                        tma_load_2d_pair(smem + i * S::kStageBytes + S::kABytes, &map_b, (kb0 + i) * kDenseBK, n0, &ctl->full[i]);
                    }
                    grid_dep_wait();
                    for (int i = 0; i < n1; ++i) tma_load_2d_pair(smem + i * S::kStageBytes, &map_a, (kb0 + i) * kDenseBK, m0, &ctl->full[i]);
                    kb = n1;
                    issued += n1;
                    s = (uint32_t)n1;
                    if (s == S::kStages) { s = 0; par ^= 1u; }
                }
                for (; kb < nkb; ++kb) {
                    if (!mbar_wait_bounded(&ctl->empty[s], par ^ 1u, &ctl->abort_flag, wait_limit_ns)) { ok = false; break; }
                    if (rank == 0) mbar_arrive_expect_tx(&ctl->full[s], 2 * S::kStageBytes);
                    uint8_t* a = smem + s * S::kStageBytes;
                    const int kx = (kb0 + kb) * kDenseBK;
                    tma_load_2d_pair(a, &map_a, kx, m0, &ctl->full[s]);
                    tma_load_2d_pair(a + S::kABytes, &map_b, kx, n0, &ctl->full[s]);
                    ++issued;
                    if (++s == S::kStages) { s = 0; par ^= 1u; }
                }
            }
            // the copies still in flight are waited for (bounded) before the pair may exit: where a wait was given up, here or later, nobody else does
            for (uint32_t back = 0; rank == 0 && back < S::kStages && back < issued; ++back) {
                if (s == 0) { s = S::kStages; par ^= 1u; }
                --s;
                if (!mbar_drain(&ctl->full[s], par, wait_limit_ns)) break;
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (rank == 0 && elect_one()) {   // one thread: lanes that a bounded wait lets go at different times could not issue together
            const uint32_t idesc = umma_idesc_bf16(256u, (uint32_t)BN);
            uint32_t s = 0, par = 0, q = 0;
            bool ok = true;
            for (int t = t0; t < ntiles && ok; t += npairs, ++q) {
                const int nkb = even_count(nkb_all, splits, t % splits);
                const uint32_t buf = q & 1u;
                ok = mbar_wait_bounded(&ctl->acc_empty[buf], ((q >> 1) & 1u) ^ 1u, &ctl->abort_flag, wait_limit_ns);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d = tmem + buf * 256u;
                for (int kb = 0; kb < nkb; ++kb) {
                    ok = mbar_wait_bounded(&ctl->full[s], par, &ctl->abort_flag, wait_limit_ns);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a = smem_u32(smem + s * S::kStageBytes);
                    const uint64_t da = umma_desc_sw128(a), db = umma_desc_sw128(a + S::kABytes);
#pragma unroll
                    for (int k4 = 0; k4 < kDenseBK / 16; ++k4)
                        umma_pair_bf16(d, da + (uint64_t)(2 * k4), db + (uint64_t)(2 * k4), idesc, (uint32_t)(kb | k4));
                    umma_commit_pair(&ctl->empty[s]);   // the slot is free, in both SMs, once these instructions have read it
                    if (++s == S::kStages) { s = 0; par ^= 1u; }
                }
                if (ok) umma_commit_pair(&ctl->acc_full[buf]);
            }
            if (!ok) {   // tensor and shared memory are given back only when no product uses them any more
                umma_commit_pair(&ctl->stopped);
                mbar_drain(&ctl->stopped, 0, wait_limit_ns);
            }
        }
        __syncwarp();
    } else {
        // epilogue: warp w reads accumulator lanes 32 * (w % 4) .. + 31 and CW of the columns; a thread owns a token row of
        // them and writes whole 32-byte sectors
        constexpr int CW = BN / kHalves;
        const int q4 = warp & 3, c0 = warp >= 6 ? CW : 0;
        uint32_t q = 0;
        float bv[kDenseTopMax];
        int bi[kDenseTopMax];
#pragma unroll
        for (int j = 0; j < kDenseTopMax; ++j) { bv[j] = -CUDART_INF_F; bi[j] = 0x7fffffff; }
        if (lane == 0) grid_dep_wait();   // the outputs may still be read by the kernels before
        __syncwarp();
        for (int t = t0; t < ntiles; t += npairs, ++q) {
            const int z = t % splits, r = t / splits, m0 = (r % mt) * 256 + (int)rank * 128, n0 = (r / mt) * BN;
            const uint32_t buf = q & 1u;
            const bool got = mbar_wait_bounded(&ctl->acc_full[buf], (q >> 1) & 1u, &ctl->abort_flag, wait_limit_ns);
            if (!__all_sync(0xffffffffu, got)) break;
            tc_fence_after();
            const uint32_t ta = tmem + buf * 256u + ((uint32_t)(q4 * 32) << 16);
            const int row = m0 + q4 * 32 + lane;
            if (EPI == EPI_PARTIAL && BN == 128) {
                // 32 x 32 sums at a time turn round in shared memory, so that a store writes four whole 128-byte lines instead of
                // 32 sectors in 32 lines (2048-token prefill at the 1.5B shape 14.72 -> 14.45 ms).  The wide tile, which the long
                // products take, gains nothing from it.
                float* turn = reinterpret_cast<float*>(smem + S::kStages * S::kStageBytes + 512) + q4 * (32 * kDenseTurnLd);
                const int r0 = m0 + q4 * 32 + lane / 8, cc = (lane % 8) * 4;
                float* dst = part + ((size_t)z * M + r0) * N + n0 + cc;
#pragma unroll 1
                for (int c = c0; c < c0 + CW; c += 32) {
                    uint32_t v[32];
                    tmem_ld32(ta + (uint32_t)c, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; i += 4)
                        *reinterpret_cast<uint4*>(turn + lane * kDenseTurnLd + i) = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                    __syncwarp();
                    if (n0 + c + cc < N) {   // N is a multiple of 16
#pragma unroll
                        for (int i = 0; i < 32; i += 4)
                            if (r0 + i < M)
                                *reinterpret_cast<float4*>(dst + (size_t)i * N + c) =
                                    *reinterpret_cast<const float4*>(turn + (i + lane / 8) * kDenseTurnLd + cc);
                    }
                    __syncwarp();
                }
            } else if (EPI == EPI_PARTIAL) {
                float* dst = part + ((size_t)z * M + row) * N + n0;
#pragma unroll 1
                for (int c = c0; c < c0 + CW; c += 32) {
                    uint32_t v[32];
                    tmem_ld32(ta + (uint32_t)c, v);
                    tmem_ld_wait();
                    if (row < M) {
#pragma unroll
                        for (int i = 0; i < 32; i += 8)
                            if (n0 + c + i < N) st_global_v8(dst + c + i, v + i);   // N is a multiple of 16
                    }
                }
            } else if (EPI == EPI_SWIGLU) {
#pragma unroll 1
                for (int c = c0; c < c0 + CW; c += 128) {
#pragma unroll 1
                    for (int e = 0; e < 64; e += 32) {
                        uint32_t g[32], u[32], pk[16];
                        tmem_ld32(ta + (uint32_t)(c + e), g);
                        tmem_ld32(ta + (uint32_t)(c + 64 + e), u);
                        tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const float g0 = __uint_as_float(g[2 * i]), g1 = __uint_as_float(g[2 * i + 1]);
                            pk[i] = pack_bf16(__fdividef(g0, 1.f + __expf(-g0)) * __uint_as_float(u[2 * i]),
                                              __fdividef(g1, 1.f + __expf(-g1)) * __uint_as_float(u[2 * i + 1]));
                        }
                        if (row < M && n0 + c < N) {
                            __nv_bfloat16* dst = out_bf16 + (size_t)row * ld_bf16 + (n0 + c) / 2 + e;
                            st_global_v8(dst, pk);
                            st_global_v8(dst + 16, pk + 8);
                        }
                    }
                }
            } else {
#pragma unroll 1
                for (int c = c0; c < c0 + CW; c += 32) {
                    uint32_t v[32];
                    tmem_ld32(ta + (uint32_t)c, v);
                    tmem_ld_wait();
                    if (n0 + c + 32 > N) {   // N is a multiple of 16
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (n0 + c + i >= N) v[i] = 0xff800000u;   // -inf
                    }
                    float m4[4];
#pragma unroll
                    for (int i = 0; i < 32; ++i) m4[i & 3] = i < 4 ? __uint_as_float(v[i]) : fmaxf(m4[i & 3], __uint_as_float(v[i]));
                    if (fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) > bv[kDenseTopMax - 1]) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) {
                            float x = __uint_as_float(v[i]);
                            // ids come in ascending order, so ">" keeps the lowest id among equals
                            if (x > bv[kDenseTopMax - 1]) {
                                int id = n0 + c + i;
#pragma unroll
                                for (int j = 0; j < kDenseTopMax; ++j)
                                    if (x > bv[j]) {
                                        const float tv = bv[j];
                                        const int ti = bi[j];
                                        bv[j] = x; bi[j] = id;
                                        x = tv; id = ti;
                                    }
                            }
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0 && t + 2 * npairs < ntiles) mbar_arrive_leader(&ctl->acc_empty[buf]);  // this warp's part of the accumulator may be overwritten
        }
        if (EPI == EPI_TOP && pair < npairs) {
            const int row = (pair % mt) * 256 + (int)rank * 128 + q4 * 32 + lane;
            if (row < M) {
                const size_t at = ((size_t)row * (kHalves * (npairs / mt)) + kHalves * (pair / mt) + (c0 != 0)) * kDenseTopMax;
                *reinterpret_cast<float4*>(top.val + at) = make_float4(bv[0], bv[1], bv[2], bv[3]);
                *reinterpret_cast<int4*>(top.idx + at) = make_int4(bi[0], bi[1], bi[2], bi[3]);
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    // Neither SM leaves while the other still reads its shared memory or signals its barriers.  Relaxed: all such accesses have been
    // waited for (every arrival above has a later product behind it), and a release would wait 0.9 us for the outputs' stores.
    cluster_arrive_relaxed();
    cluster_wait();
    tc_fence_after();
    if (warp == 1) tmem_dealloc_pair(tmem, 512);
    if (threadIdx.x == 0 && ctl->abort_flag) atomicExch(err, 1);
}

// Sum over a block of up to 1024 threads, handed to every thread.
__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    v = (threadIdx.x & 31) < (blockDim.x >> 5) ? red[threadIdx.x & 31] : 0.f;
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Residual rows: h[r] = embedding of token r (tokens != nullptr) or h[r] + the K shares' partial sums of the
// product before; then the norm of the next product: xn[r] = bf16(h[r] * rsqrt(mean(h[r]^2) + eps) * w).  One block
// per row, four columns per thread (d > 4096: several turns); the row is read once, sums and norm stay in registers.
// h_last: a copy of the last row (or nullptr).  Bound by the launch and one L2 round trip (a few MB).  T: turns kept in
// registers.  One or two turns (d <= 4096) take blocks of up to 512 threads, two of which fit an SM, so that 256 rows are
// resident at once (7B shape: 7.2 -> 5.2 us a launch; 1.5B 4.1 -> 3.9).
template <int T>
__global__ void __launch_bounds__(T <= 2 ? 512 : 1024, T <= 2 ? 2 : 1)
dense_residual_norm_kernel(const int* tokens, const __nv_bfloat16* emb, int V, float* h, const float* part, int splits, const float* w,
                           __nv_bfloat16* xn, int d, float eps, float* h_last) {
    __shared__ float red[32];
    const int row = blockIdx.x, n4 = d / 4;
    grid_dep_launch();
    float4 v[T], g[T];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        const int c = threadIdx.x + t * blockDim.x;
        g[t] = c < n4 ? __ldg(reinterpret_cast<const float4*>(w) + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        asm volatile("" ::"f"(g[t].x), "f"(g[t].y), "f"(g[t].z), "f"(g[t].w));   // asked for here, while the product still runs
    }
    grid_dep_wait();
    float* hr = h + (size_t)row * d;
    float ss = 0.f;
#pragma unroll
    for (int t = 0; t < T; ++t) {
        const int c = threadIdx.x + t * blockDim.x;
        if (c < n4) {
            float4 x;
            if (tokens) {
                const int tok = min(max(tokens[row], 0), V - 1);
                const uint2 raw = *reinterpret_cast<const uint2*>(emb + (size_t)tok * d + c * 4);
                const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x));
                const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
                x = make_float4(a.x, a.y, b.x, b.y);
            } else {
                x = reinterpret_cast<const float4*>(hr)[c];
                const float4* p = reinterpret_cast<const float4*>(part + (size_t)row * d) + c;
                const size_t stride = (size_t)gridDim.x * n4;
#pragma unroll 4
                for (int z = 0; z < splits; ++z) {
                    const float4 y = __ldcg(p + z * stride);
                    x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
                }
            }
            reinterpret_cast<float4*>(hr)[c] = x;
            if (h_last && row == (int)gridDim.x - 1) reinterpret_cast<float4*>(h_last)[c] = x;
            ss += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
            v[t] = x;
        }
    }
    const float rs = rsqrtf(block_sum(ss, red) / (float)d + eps);
#pragma unroll
    for (int t = 0; t < T; ++t) {
        const int c = threadIdx.x + t * blockDim.x;
        if (c < n4)
            *reinterpret_cast<uint2*>(xn + (size_t)row * d + c * 4) =
                make_uint2(pack_bf16(v[t].x * rs * g[t].x, v[t].y * rs * g[t].y), pack_bf16(v[t].z * rs * g[t].z, v[t].w * rs * g[t].w));
    }
}

// q|k|v of a row: sums over the K shares, bias, rotary embedding of q and k at position L + r (pairing (i, i + hd/2));
// q to the bf16 query matrix, k and v appended to the cache.  One block per row, four rotary pairs per thread and turn.
// Bound like the one above; bias and rotary factors are fetched while the product still runs, and a block holds the row in
// one turn (7B shape: 5.3 -> 2.6 us a launch, 1.5B 3.2 -> 2.6).
__global__ void __launch_bounds__(1024) dense_qkv_finish_kernel(const float* part, int splits, const float* bias, const float2* rope,
                                                               __nv_bfloat16* qout, int n_q, int n_kv, int hd, __nv_bfloat16* kcache,
                                                               __nv_bfloat16* vcache, size_t layer_off, int max_seq, int L) {
    const int r = blockIdx.x, h2 = hd / 2, per_head = h2 / 4, n_qkv = (n_q + 2 * n_kv) * hd;
    const size_t stride = (size_t)gridDim.x * n_qkv;
    grid_dep_launch();
    for (int it = threadIdx.x; it < (n_q + 2 * n_kv) * per_head; it += blockDim.x) {
        const int head = it / per_head, i = (it % per_head) * 4;
        const float* p = part + (size_t)r * n_qkv + head * hd + i;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (bias) {
            a = __ldg(reinterpret_cast<const float4*>(bias + head * hd + i));
            b = __ldg(reinterpret_cast<const float4*>(bias + head * hd + i + h2));
        }
        const float4* cs = reinterpret_cast<const float4*>(rope + (size_t)(L + r) * h2 + i);
        const float4 c0 = __ldg(cs), c1 = __ldg(cs + 1);
        if (it == (int)threadIdx.x) grid_dep_wait();
#pragma unroll 4
        for (int z = 0; z < splits; ++z) {
            const float4 x = __ldcg(reinterpret_cast<const float4*>(p + z * stride));
            const float4 y = __ldcg(reinterpret_cast<const float4*>(p + z * stride + h2));
            a.x += x.x; a.y += x.y; a.z += x.z; a.w += x.w;
            b.x += y.x; b.y += y.y; b.z += y.z; b.w += y.w;
        }
        __nv_bfloat16* dst;
        if (head < n_q) dst = qout + (size_t)r * (n_q * hd) + head * hd;
        else if (head < n_q + n_kv) dst = kcache + layer_off + ((size_t)(head - n_q) * max_seq + L + r) * hd;
        else dst = vcache + layer_off + ((size_t)(head - n_q - n_kv) * max_seq + L + r) * hd;
        float4 lo = a, hi = b;
        if (head < n_q + n_kv) {
            lo = make_float4(a.x * c0.x - b.x * c0.y, a.y * c0.z - b.y * c0.w, a.z * c1.x - b.z * c1.y, a.w * c1.z - b.w * c1.w);
            hi = make_float4(b.x * c0.x + a.x * c0.y, b.y * c0.z + a.y * c0.w, b.z * c1.x + a.z * c1.y, b.w * c1.z + a.w * c1.w);
        }
        *reinterpret_cast<uint2*>(dst + i) = make_uint2(pack_bf16(lo.x, lo.y), pack_bf16(lo.z, lo.w));
        *reinterpret_cast<uint2*>(dst + i + h2) = make_uint2(pack_bf16(hi.x, hi.y), pack_bf16(hi.z, hi.w));
    }
}

// Causal attention of a sub-chunk's queries (rows r = 0..M-1 at positions L + r) over cache rows 0 .. L + r of their
// KV head.  A block's 128 tile rows are the queries of all g heads that share a KV head: tile row t = query q0 + t / g, head
// t % g.  The keys are cut into contiguous shares over the blocks of a cluster, a share into blocks of 128 keys (tensor-map
// copies into a ring).  Even and odd key blocks are two independent streams, each with its own scores S, output O
// and running maximum in tensor memory and a warpgroup of its own (one tile row per thread): while one warpgroup
// turns its scores into probabilities (written back over S as bf16, the A operand of P V), the tensor core works for the
// other.  O is rescaled only when the maximum grew by more than 2^8 (the probabilities then stay below 2^8, the sums
// are fp32).  The two alternating streams with P in tensor memory and the rare rescaling are the method published as
// FlashAttention-4; grouped heads as tile rows, keys over a cluster and the exchange are this kernel's.  The blocks of a cluster merge their rows by bulk copies between their shared memories: each finishes an
// even share of the tile rows and is sent the others' outputs of them, with maximum and sum behind every row.  (Reading
// them by remote loads took 4 to 6 us of a launch, 13 bytes per cycle and SM.)  Output bf16 [M][n_q * hd].
// Bound by the exponentials (16 per cycle and SM: 1.1 us per 128 keys of both streams) and, over short contexts, by the
// chain load -> S -> softmax -> P V -> merge.  Mean over the eight 256-token chunks of a 2048-token request at the 1.5B
// shape: 11.5 us a launch (14.3 with remote loads, 35 with mma.sync tiles); 7B 14.2 us (18.5).
template <int HD>
struct DenseAttShape {
    static constexpr int kAtoms = HD / 64;                       // 64-column swizzled slabs of a row
    static constexpr int kTileBytes = 128 * HD * 2;              // queries, or the keys or values of a block
    static constexpr int kStages = 3;
    static constexpr int kLdo = HD + 4;                          // floats of an exchanged row: output, maximum in log2 units, sum, padding
    static constexpr int kExBytes = 128 * kLdo * 4;              // the block's outputs
    static constexpr int kRing = kStages * 2 * kTileBytes;
    static constexpr int kInBytes = (128 + 8) * kLdo * 4;        // the other blocks' outputs for this block's rows (up to eight shares, rounded up)
    static constexpr int kSmemBytes = kTileBytes + kRing + 256 + 1024;
    static_assert(kExBytes + kInBytes <= kRing, "the exchange areas reuse the ring");
};
constexpr int kDenseAttThreads = 320;   // warps 0..3 and 4..7: the two streams; 8: copies; 9: tensor-core issue

template <int HD>
__global__ void __launch_bounds__(kDenseAttThreads, 1)
dense_attention_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const __nv_bfloat16* q,
                       int cache_row0, int max_seq, int n_q, int g, int QR, int M, int L, float scale_log2e, __nv_bfloat16* out,
                       int* err, unsigned long long wait_limit_ns) {
    using S = DenseAttShape<HD>;
    constexpr int KSTEPS = HD / 16, UNITS = HD / 8;
    extern __shared__ uint8_t att_smem_raw[];
    uint8_t* Qs = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(att_smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* ring = Qs + S::kTileBytes;                                  // [stage][K | V]
    float2* ex_ml = reinterpret_cast<float2*>(Qs);   // once the products are done: [stream][tile row] (maximum in log2 units, sum)
    struct Ctl {
        uint64_t kfull[S::kStages], vfull[S::kStages], empty[S::kStages], s_full[2], p_ready[2], o_full, in_full;
        uint32_t tmem_base;
        int abort_flag;
    };
    Ctl* ctl = reinterpret_cast<Ctl*>(ring + S::kRing);
    static_assert(sizeof(Ctl) <= 256, "control block");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
    const int CS = (int)cluster_size(), rank = (int)cluster_rank();
    const int kvh = blockIdx.y, q0 = ((int)blockIdx.x / CS) * QR;       // first query of the block
    const int nkeys = L + min(M, q0 + QR);                              // keys any row of this block may see
    const int nblk_all = (nkeys + 127) / 128;
    const int b0 = even_start(nblk_all, CS, rank), nblk = even_count(nblk_all, CS, rank);
    const int R = min(QR, M - q0) * g, rbeg = even_start(R, CS, rank), rows = even_count(R, CS, rank);   // tile rows; those this block finishes
    if (tid == 0) {
        for (int s = 0; s < S::kStages; ++s) {
            mbar_init(&ctl->kfull[s], 1);
            mbar_init(&ctl->vfull[s], 1);
            mbar_init(&ctl->empty[s], 1);
        }
        for (int w = 0; w < 2; ++w) {
            mbar_init(&ctl->s_full[w], 1);
            mbar_init(&ctl->p_ready[w], 4);
        }
        mbar_init(&ctl->o_full, 1);
        mbar_init(&ctl->in_full, 1);
        ctl->abort_flag = 0;
        mbar_fence_init();
        mbar_arrive_expect_tx(&ctl->in_full, (uint32_t)((CS - 1) * rows * S::kLdo * 4));
    }
    if (warp == 9) tmem_alloc(&ctl->tmem_base, 512);   // S0 | S1 | O0 | O1, 128 columns each
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    grid_dep_launch();
    constexpr int QI = 128 * UNITS / 256;   // 16-byte units of the query tile per thread
    int qoff[QI];                           // where they are, -1: a row without a query (worked out while the kernel before runs)
#pragma unroll
    for (int i = 0; i < QI; ++i) {
        const int u = tid + i * 256, t = u / UNITS, qi = q0 + t / g;
        qoff[i] = t < QR * g && qi < M ? qi * (n_q * HD) + (kvh * g + t % g) * HD + (u % UNITS) * 8 : -1;
    }
    grid_dep_wait();
    if (warp < 8) {
        // query tile, in the layout the copies have: slabs of 64 columns, 128-byte swizzle; all loads in flight
        uint4 v[QI];
#pragma unroll
        for (int i = 0; i < QI; ++i) v[i] = qoff[i] < 0 ? make_uint4(0, 0, 0, 0) : __ldcg(reinterpret_cast<const uint4*>(q + qoff[i]));
#pragma unroll
        for (int i = 0; i < QI; ++i) {
            const int u = tid + i * 256, c16 = u % UNITS;
            *reinterpret_cast<uint4*>(Qs + (c16 >> 3) * 16384 + swz_unit(u / UNITS, c16 & 7)) = v[i];
        }
    }
    if (warp != 8) {
        fence_proxy_async_smem();
        named_bar_sync(2, 288);   // the queries are in place for the tensor-core warp
    }

    if (warp == 8) {
        if (elect_one()) {
            uint32_t s = 0, par = 0;
            int issued = 0;
            const int y0 = cache_row0 + kvh * max_seq + b0 * 128;
            for (; issued < nblk; ++issued) {
                if (!mbar_wait_bounded(&ctl->empty[s], par ^ 1u, &ctl->abort_flag, wait_limit_ns)) break;
                uint8_t* ks = ring + s * 2 * S::kTileBytes;
                const int y = y0 + issued * 128;
                mbar_arrive_expect_tx(&ctl->kfull[s], S::kTileBytes);
                for (int a = 0; a < S::kAtoms; ++a) tma_load_2d(ks + a * 16384, &map_k, a * 64, y, &ctl->kfull[s]);
                mbar_arrive_expect_tx(&ctl->vfull[s], S::kTileBytes);
                for (int a = 0; a < S::kAtoms; ++a) tma_load_2d(ks + S::kTileBytes + a * 16384, &map_v, a * 64, y, &ctl->vfull[s]);
                if (++s == S::kStages) { s = 0; par ^= 1u; }
            }
            // the copies still in flight are waited for (bounded): where a wait was given up, here or later, nobody else does
            for (int back = 0; back < S::kStages && back < issued; ++back) {
                if (s == 0) { s = S::kStages; par ^= 1u; }
                --s;
                if (!(mbar_drain(&ctl->kfull[s], par, wait_limit_ns) && mbar_drain(&ctl->vfull[s], par, wait_limit_ns))) break;
            }
        }
        __syncwarp();
    } else if (warp == 9) {
        const uint32_t id_s = umma_idesc_bf16(128u, 128u), id_o = umma_idesc_bf16(128u, (uint32_t)HD) | (1u << 16);   // B of P V: features contiguous
        bool ok = true;
        auto scores = [&](int j) {
            const int s = j % S::kStages;
            ok = ok && mbar_wait_bounded(&ctl->kfull[s], (uint32_t)(j / S::kStages) & 1u, &ctl->abort_flag, wait_limit_ns);
            if (!__all_sync(0xffffffffu, ok)) { ok = false; return; }
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(j & 1) * 128u, k = smem_u32(ring + s * 2 * S::kTileBytes), qa = smem_u32(Qs);
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < KSTEPS; ++ks) {
                    const uint32_t off = (uint32_t)((ks >> 2) * 16384 + (ks & 3) * 32);
                    umma_bf16(d, umma_desc_sw128(qa + off), umma_desc_sw128(k + off), id_s, (uint32_t)ks);
                }
                umma_commit(&ctl->s_full[j & 1]);
            }
            __syncwarp();
        };
        if (nblk > 0) scores(0);
        if (nblk > 1) scores(1);
        for (int j = 0; j < nblk && ok; ++j) {
            const int s = j % S::kStages, w = j & 1;
            ok = mbar_wait_bounded(&ctl->vfull[s], (uint32_t)(j / S::kStages) & 1u, &ctl->abort_flag, wait_limit_ns) &&
                 mbar_wait_bounded(&ctl->p_ready[w], (uint32_t)(j >> 1) & 1u, &ctl->abort_flag, wait_limit_ns);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const uint32_t v = smem_u32(ring + s * 2 * S::kTileBytes + S::kTileBytes);
            if (elect_one()) {
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)   // 16 keys: 16 rows of 128 bytes of every slab; 8 packed columns of P
                    umma_bf16_tmem_a(tmem + 256u + (uint32_t)w * 128u, tmem + (uint32_t)w * 128u + (uint32_t)ks * 8u,
                                     umma_desc_sw128_mn(v + (uint32_t)ks * 2048u, 16384u), id_o, (uint32_t)((j >> 1) | ks));
                umma_commit(&ctl->empty[s]);
            }
            __syncwarp();
            if (j + 2 < nblk) scores(j + 2);
        }
        // behind an abandoned wait as well: tensor and shared memory are given back only when no product uses them any more
        if (elect_one()) umma_commit(&ctl->o_full);
        __syncwarp();
        if (!ok) mbar_drain(&ctl->o_full, 0, wait_limit_ns);
    } else {
        const int w = warp >> 2, t = (warp & 3) * 32 + lane;   // stream, tile row
        const uint32_t ts = tmem + (uint32_t)w * 128u + ((uint32_t)((warp & 3) * 32) << 16), to = ts + 256u;
        const int lim = L + q0 + t / g;                        // last key this row sees
        float m = -CUDART_INF_F, l = 0.f;
        bool ok = true;
        for (int j = w; j < nblk; j += 2) {
            const int s = j % S::kStages, key0 = (b0 + j) * 128;
            ok = ok && mbar_wait_bounded(&ctl->s_full[w], (uint32_t)(j >> 1) & 1u, &ctl->abort_flag, wait_limit_ns);
            if (key0 + 128 > nkeys) {
                // values behind the last key are whatever the cache holds there: cleared, since 0 x NaN is not 0
                ok = ok && mbar_wait_bounded(&ctl->vfull[s], (uint32_t)(j / S::kStages) & 1u, &ctl->abort_flag, wait_limit_ns);
                if (ok && key0 + t >= nkeys) {
                    uint4* vr = reinterpret_cast<uint4*>(ring + s * 2 * S::kTileBytes + S::kTileBytes + t * 128);
#pragma unroll
                    for (int i = 0; i < UNITS; ++i) vr[(i >> 3) * 1024 + (i & 7)] = make_uint4(0, 0, 0, 0);
                }
                fence_proxy_async_smem();
            }
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const int seen = lim - key0;                       // columns 0..seen are visible
            uint32_t v[4][32];   // the row's 128 scores, read once
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld32(ts + 32u * (uint32_t)c, v[c]);
            tmem_ld_wait();
            if (seen < 127) {
#pragma unroll
                for (int i = 0; i < 128; ++i)
                    if (i > seen) v[i >> 5][i & 31] = 0xff800000u;   // -inf
            }
            float m4[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};   // four independent chains
#pragma unroll
            for (int i = 0; i < 128; ++i) m4[i & 3] = fmaxf(m4[i & 3], __uint_as_float(v[i >> 5][i & 31]));
            float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
            mx *= scale_log2e;
            const bool grow = mx > m + 8.f;                    // also the first block that shows this row a key
            if (__any_sync(0xffffffffu, grow && m != -CUDART_INF_F)) {
                const float f = grow && m != -CUDART_INF_F ? exp2f(m - mx) : 1.f;
                l *= f;
#pragma unroll 1
                for (int c = 0; c < HD; c += 16) {
                    float o[16];
                    uint32_t u[16];
                    tmem_ld16(to + (uint32_t)c, o);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 16; ++i) u[i] = __float_as_uint(o[i] * f);
                    tmem_st16(to + (uint32_t)c, u);
                }
            }
            if (grow) m = mx;
            const float ref = m == -CUDART_INF_F ? 0.f : m;
            float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t pk[16];
#pragma unroll
                for (int i = 0; i < 32; i += 2) {
                    const float x = ex2_ftz(fmaf(__uint_as_float(v[c][i]), scale_log2e, -ref));
                    const float y = ex2_ftz(fmaf(__uint_as_float(v[c][i + 1]), scale_log2e, -ref));
                    s4[i & 2] += x;
                    s4[(i & 2) + 1] += y;
                    pk[i / 2] = pack_bf16(x, y);
                }
                tmem_st16(ts + 16u * (uint32_t)c, pk);         // over scores this thread has read
            }
            const float sum = (s4[0] + s4[1]) + (s4[2] + s4[3]);
            l += sum;
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->p_ready[w]);
        }
        // The two streams of a row meet: statistics through shared memory, outputs straight from tensor memory (each
        // warpgroup takes half of the columns).  The ring and the queries are free once every product has completed.
        if (nblk > 0) ok = ok && mbar_wait_bounded(&ctl->o_full, 0, &ctl->abort_flag, wait_limit_ns);
        ok = __all_sync(0xffffffffu, ok);
        ex_ml[w * 128 + t] = ok ? make_float2(m, l) : make_float2(-CUDART_INF_F, 0.f);
        named_bar_sync(1, 256);
        if (CS > 1) cluster_arrive();   // nothing reads this block's ring any more
        const float2 o0 = ex_ml[t], o1 = ex_ml[128 + t];
        const float mx = fmaxf(o0.x, o1.x), ref = mx == -CUDART_INF_F ? 0.f : mx;
        const float w0 = exp2f(o0.x - ref), w1 = exp2f(o1.x - ref);
        const float sum = w0 * o0.y + w1 * o1.y;
        const float sc = CS == 1 ? 1.f / sum : 1.f;   // a block that saw all keys writes the result itself
        const int qi = q0 + t / g;
        __nv_bfloat16* po = out + (size_t)qi * (n_q * HD) + (kvh * g + t % g) * HD;
        float* ex = reinterpret_cast<float*>(ring) + t * S::kLdo;
        if (w == 0 && CS > 1) *reinterpret_cast<float2*>(ex + HD) = make_float2(mx, sum);
        if (nblk > 0 && ok) {
            tc_fence_after();
#pragma unroll 1
            for (int c = w * (HD / 2); c < (w + 1) * (HD / 2); c += 32) {
                uint32_t a[32], b[32];
                tmem_ld32(tmem + 256u + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c, a);
                tmem_ld32(tmem + 384u + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c, b);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 32; i += 4) {
                    float4 v = make_float4(w0 * __uint_as_float(a[i]), w0 * __uint_as_float(a[i + 1]), w0 * __uint_as_float(a[i + 2]),
                                           w0 * __uint_as_float(a[i + 3]));
                    if (nblk > 1) {   // the second stream wrote its output
                        v.x += w1 * __uint_as_float(b[i]); v.y += w1 * __uint_as_float(b[i + 1]);
                        v.z += w1 * __uint_as_float(b[i + 2]); v.w += w1 * __uint_as_float(b[i + 3]);
                    }
                    if (CS > 1) *reinterpret_cast<float4*>(ex + c + i) = v;
                    else if (t < QR * g && qi < M)
                        *reinterpret_cast<uint2*>(po + c + i) = make_uint2(pack_bf16(v.x * sc, v.y * sc), pack_bf16(v.z * sc, v.w * sc));
                }
            }
        }
        tc_fence_before();
        fence_proxy_async_smem();
    }
    __syncwarp();
    if (CS > 1) {
        if (warp >= 8) cluster_arrive();
        cluster_wait();
    }
    __syncthreads();
    if (warp == 9) tmem_dealloc(tmem, 512);
    if (CS == 1) {
        if (tid == 0 && ctl->abort_flag) atomicExch(err, 1);
        return;
    }
    // every block finishes its share of the tile rows: the others send it their outputs and statistics of them
    const uint32_t ex = smem_u32(ring), in = ex + S::kExBytes;
    constexpr uint32_t kRowBytes = S::kLdo * 4;
    if (tid < CS && tid != rank) {
        const int n = even_count(R, CS, tid);
        if (n) bulk_s2cluster(map_shared_rank(in + (uint32_t)(rank * n) * kRowBytes, tid), ex + (uint32_t)even_start(R, CS, tid) * kRowBytes,
                              (uint32_t)n * kRowBytes, map_shared_rank(smem_u32(&ctl->in_full), tid));
    }
    __syncwarp();
    const bool got = mbar_wait_bounded(&ctl->in_full, 0, &ctl->abort_flag, wait_limit_ns);
    if (!got) mbar_drain(&ctl->in_full, 0, wait_limit_ns);   // a wait was given up, but the others send all the same: not into a block that has left
    __syncwarp();
    cluster_arrive();   // what was sent to this block has left its senders
    if (got) {
        constexpr int C8 = HD / 8;
        for (int it = tid; it < rows * C8; it += kDenseAttThreads) {
            const int i = it / C8, t = rbeg + i, c = (it % C8) * 8;
            auto part = [&](int k) {
                return reinterpret_cast<const float*>(k == rank ? ring + t * kRowBytes : ring + S::kExBytes + (k * rows + i) * kRowBytes);
            };
            float mx = -CUDART_INF_F, sum = 0.f;
            for (int k = 0; k < CS; ++k) mx = fmaxf(mx, part(k)[HD]);
            float o[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            for (int k = 0; k < CS; ++k) {
                const float* p = part(k);
                if (p[HD] == -CUDART_INF_F) continue;   // a block without a key never wrote its outputs
                const float w = exp2f(p[HD] - mx);
                const float4 x = *reinterpret_cast<const float4*>(p + c), y = *reinterpret_cast<const float4*>(p + c + 4);
                sum += w * p[HD + 1];
                o[0] += w * x.x; o[1] += w * x.y; o[2] += w * x.z; o[3] += w * x.w;
                o[4] += w * y.x; o[5] += w * y.y; o[6] += w * y.z; o[7] += w * y.w;
            }
            const float sc = 1.f / sum;
            *reinterpret_cast<uint4*>(out + (size_t)(q0 + t / g) * (n_q * HD) + (kvh * g + t % g) * HD + c) =
                make_uint4(pack_bf16(o[0] * sc, o[1] * sc), pack_bf16(o[2] * sc, o[3] * sc), pack_bf16(o[4] * sc, o[5] * sc), pack_bf16(o[6] * sc, o[7] * sc));
        }
    }
    __syncwarp();
    cluster_wait();   // and what this block sent has left
    if (tid == 0 && ctl->abort_flag) atomicExch(err, 1);
}

// Calibration, "Sample": the b best ids of every row from the shares' best kDenseTopMax (largest first, lowest id among
// equals).  One block per row.
__global__ void __launch_bounds__(256) dense_top_merge_kernel(DenseTopOut top, int shares, int b, int* succ /* [rows][b] */) {
    __shared__ float bv_s[8];
    __shared__ int bi_s[8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n = shares * kDenseTopMax;
    grid_dep_launch();
    grid_dep_wait();
    const float* val = top.val + (size_t)blockIdx.x * n;
    const int* idx = top.idx + (size_t)blockIdx.x * n;
    float last_v = CUDART_INF_F;
    int last_i = -1;   // the winner before: later ones come behind it in (value descending, id ascending) order
    for (int r = 0; r < b; ++r) {
        float bv = -CUDART_INF_F;
        int bi = 0x7fffffff;
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const float v = val[i];
            const int id = idx[i];
            const bool behind = v < last_v || (v == last_v && id > last_i);
            if (behind && (v > bv || (v == bv && id < bi))) { bv = v; bi = id; }
        }
#pragma unroll
        for (int off = 16; off; off >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, off);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
            if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
        }
        __syncthreads();
        if (lane == 0) { bv_s[warp] = bv; bi_s[warp] = bi; }
        __syncthreads();
        bv = bv_s[0];
        bi = bi_s[0];
        for (int w = 1; w < 8; ++w)
            if (bv_s[w] > bv || (bv_s[w] == bv && bi_s[w] < bi)) { bv = bv_s[w]; bi = bi_s[w]; }
        last_v = bv;
        last_i = bi;
        if (threadIdx.x == 0) succ[(size_t)blockIdx.x * b + r] = bi == 0x7fffffff ? 0 : bi;
    }
}

// Weight copy for the dense path.  mode 0: rows copied as they are (dst row = src row).  mode 1:
// gate | up interleaved in blocks of 64: dst rows [128 t, 128 t + 64) = gate rows 64 t.., the next 64
// rows the matching up rows, so that 128 columns of a tile hold both halves of 64 SwiGLU columns.
__global__ void dense_copy_weights_kernel(uint16_t* dst, const uint16_t* src0, const uint16_t* src1, int rows, int K, int mode) {
    const int K8 = K / 8;
    const long long total = (long long)rows * K8;
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < total; u += (long long)gridDim.x * blockDim.x) {
        const int r = (int)(u / K8), k8 = (int)(u % K8);
        const uint16_t* s;
        if (mode == 0) {
            s = src0 + (size_t)r * K;
        } else {
            const int t = r / 128, w = r % 128;
            s = (w < 64) ? src0 + (size_t)(64 * t + w) * K : src1 + (size_t)(64 * t + w - 64) * K;
        }
        *reinterpret_cast<uint4*>(dst + (size_t)r * K + k8 * 8) = *reinterpret_cast<const uint4*>(s + k8 * 8);
    }
}

}  // namespace sdv
