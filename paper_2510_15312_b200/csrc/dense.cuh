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
constexpr int kDenseThreads = 192;      // warp 0: copies, warp 1: tensor-core issue, warps 2..5: epilogue
constexpr int kDenseMaxRows = 1024;     // rows of the activation buffers (one sub-chunk)
constexpr int kDenseMaxSplits = 16;     // K shares of one product at most
constexpr int kDenseTopMax = 4;         // best logits kept per row and vocabulary tile (calibration)

enum DenseEpilogue { EPI_PARTIAL = 0, EPI_SWIGLU = 1, EPI_TOP = 2 };

// Stage of a pair tile of 256 tokens x BN features: every SM of the pair holds 128 token rows and half of the
// features' weight rows.
template <int BN>
struct DenseShape {
    static constexpr int kABytes = 128 * kDenseBK * 2;
    static constexpr int kBBytes = BN / 2 * kDenseBK * 2;
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kStages = BN == 256 ? 6 : 8;
    static constexpr int kSmemBytes = kStages * kStageBytes + 1024 + 512;
};

// Shared-memory operand descriptor, K-major, 128-byte swizzle: rows of 64 bf16 (128 bytes), groups of
// 8 rows 1024 bytes apart; a 16-element K step advances the start address by 32 bytes.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3fffu);
    d |= (uint64_t)1 << 16;                         // leading byte offset: unused for swizzled K-major operands
    d |= (uint64_t)(1024u >> 4) << 32;              // stride between 8-row groups
    d |= (uint64_t)1 << 46;                         // descriptor version of this architecture
    d |= (uint64_t)2 << 61;                         // 128-byte swizzle
    return d;
}

struct DenseTopOut {   // EPI_TOP: [row][vocabulary tile][kDenseTopMax] best logits of the tile and their ids, best first
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
//   EPI_TOP:     the best kDenseTopMax values of every row in this tile of features (largest first, lowest id first
//                among equals)
// Rows >= M and columns >= N are computed on whatever the copies deliver (zeros outside the tensors) and
// never written.  err: set to 1 when a bounded wait runs out.
// Measured on B200 (BN 256, 1536 x 17920 weights): 256 tokens 18.6 us stand-alone (758 TFLOP/s; 25.4 us with
// 128 x 128 tiles on single SMs), 1024 tokens 41 us (1371 TFLOP/s).  With 256 tokens the weights' HBM read
// (8.4 us) and the fill and drain of the pipeline bound it, with 1024 the tensor cores.
template <int EPI, int BN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kDenseThreads, 1)
dense_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b, int M, int N, int K,
                  int splits, float* part, __nv_bfloat16* out_bf16, int ld_bf16, DenseTopOut top, int* err,
                  unsigned long long wait_limit_ns) {
    using S = DenseShape<BN>;
    extern __shared__ uint8_t dense_smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dense_smem_raw) + 1023) & ~(uintptr_t)1023);
    struct Ctl {
        uint64_t full[S::kStages], empty[S::kStages];  // full: the leading SM's counts both SMs' bytes
        uint64_t acc_full[2], acc_empty[2];            // acc_empty: the leading SM's counts both SMs' epilogue warps
        uint32_t tmem_base;
        int abort_flag;
    };
    Ctl* ctl = reinterpret_cast<Ctl*>(smem + S::kStages * S::kStageBytes);
    static_assert(sizeof(Ctl) <= 512, "control block");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int mt = (M + 255) / 256, nt = (N + BN - 1) / BN, ntiles = mt * nt * splits;
    const int nkb_all = K / kDenseBK;
    const int npairs = (int)gridDim.x >> 1, pair = (int)blockIdx.x >> 1;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S::kStages; ++s) {
            mbar_init(&ctl->full[s], 1);
            mbar_init(&ctl->empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&ctl->acc_full[b], 1);
            mbar_init(&ctl->acc_empty[b], 8);
        }
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
            for (int t = pair; t < ntiles && ok; t += npairs) {
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
            if (!ok && rank == 0) {
                // abandoned: wait (bounded) for the copies still in flight before the pair may exit
                for (uint32_t back = 0; back < S::kStages && back < issued; ++back) {
                    if (s == 0) { s = S::kStages; par ^= 1u; }
                    --s;
                    const uint64_t t0 = global_timer_ns();
                    while (!mbar_try_wait(&ctl->full[s], par) && global_timer_ns() - t0 < wait_limit_ns) {}
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (rank == 0) {
            const uint32_t idesc = umma_idesc_bf16(256u, (uint32_t)BN);
            uint32_t s = 0, par = 0, q = 0;
            bool ok = true;
            for (int t = pair; t < ntiles && ok; t += npairs, ++q) {
                const int nkb = even_count(nkb_all, splits, t % splits);
                const uint32_t buf = q & 1u;
                if (!mbar_wait_bounded(&ctl->acc_empty[buf], ((q >> 1) & 1u) ^ 1u, &ctl->abort_flag, wait_limit_ns)) break;
                tc_fence_after();
                const uint32_t d = tmem + buf * 256u;
                for (int kb = 0; kb < nkb; ++kb) {
                    ok = mbar_wait_bounded(&ctl->full[s], par, &ctl->abort_flag, wait_limit_ns);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a = smem_u32(smem + s * S::kStageBytes);
                    const uint64_t da = umma_desc_sw128(a), db = umma_desc_sw128(a + S::kABytes);
                    if (elect_one()) {
#pragma unroll
                        for (int k4 = 0; k4 < kDenseBK / 16; ++k4)
                            umma_pair_bf16(d, da + (uint64_t)(2 * k4), db + (uint64_t)(2 * k4), idesc, (uint32_t)(kb | k4));
                        umma_commit_pair(&ctl->empty[s]);   // the slot is free, in both SMs, once these instructions have read it
                    }
                    __syncwarp();
                    if (++s == S::kStages) { s = 0; par ^= 1u; }
                }
                if (ok && elect_one()) umma_commit_pair(&ctl->acc_full[buf]);
                __syncwarp();
            }
        }
    } else {
        // epilogue: warp w reads accumulator lanes 32 * (w % 4) .. + 31; a thread owns one token row of the tile and
        // writes whole 32-byte sectors of it
        const int q4 = warp & 3;
        uint32_t q = 0;
        if (lane == 0) grid_dep_wait();   // the outputs may still be read by the kernels before
        __syncwarp();
        for (int t = pair; t < ntiles; t += npairs, ++q) {
            const int z = t % splits, r = t / splits, m0 = (r % mt) * 256 + (int)rank * 128, n0 = (r / mt) * BN;
            const uint32_t buf = q & 1u;
            const bool got = mbar_wait_bounded(&ctl->acc_full[buf], (q >> 1) & 1u, &ctl->abort_flag, wait_limit_ns);
            if (!__all_sync(0xffffffffu, got)) break;
            tc_fence_after();
            const uint32_t ta = tmem + buf * 256u + ((uint32_t)(q4 * 32) << 16);
            const int row = m0 + q4 * 32 + lane;
            if (EPI == EPI_PARTIAL) {
                float* dst = part + ((size_t)z * M + row) * N + n0;
#pragma unroll 1
                for (int c = 0; c < BN; c += 32) {
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
                for (int c = 0; c < BN; c += 128) {
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
                float bv[kDenseTopMax];
                int bi[kDenseTopMax];
#pragma unroll
                for (int j = 0; j < kDenseTopMax; ++j) { bv[j] = -CUDART_INF_F; bi[j] = 0x7fffffff; }
#pragma unroll 1
                for (int c = 0; c < BN; c += 32) {
                    uint32_t v[32];
                    tmem_ld32(ta + (uint32_t)c, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        float x = __uint_as_float(v[i]);
                        // ids come in ascending order, so ">" keeps the lowest id among equals
                        if (x > bv[kDenseTopMax - 1] && n0 + c + i < N) {
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
                if (row < M) {
                    const size_t at = ((size_t)row * nt + r / mt) * kDenseTopMax;
                    *reinterpret_cast<float4*>(top.val + at) = make_float4(bv[0], bv[1], bv[2], bv[3]);
                    *reinterpret_cast<int4*>(top.idx + at) = make_int4(bi[0], bi[1], bi[2], bi[3]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_leader(&ctl->acc_empty[buf]);  // this warp's part of the accumulator may be overwritten
        }
    }
    __syncwarp();
    tc_fence_before();
    cluster_sync();   // neither SM leaves while the other still reads its shared memory or signals its barriers
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
// h_last: a copy of the last row (or nullptr).  Bound by the launch and one L2 round trip (a few MB).
__global__ void __launch_bounds__(1024) dense_residual_norm_kernel(const int* tokens, const __nv_bfloat16* emb, int V, float* h,
                                                                    const float* part, int splits, const float* w,
                                                                    __nv_bfloat16* xn, int d, float eps, float* h_last) {
    __shared__ float red[32];
    const int row = blockIdx.x, n4 = d / 4;
    grid_dep_launch();
    constexpr int T = 4;   // turns kept in registers: d <= 16384
    float4 v[T], g[T];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        const int c = threadIdx.x + t * blockDim.x;
        if (c < n4) g[t] = __ldg(reinterpret_cast<const float4*>(w) + c);
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
__global__ void __launch_bounds__(256) dense_qkv_finish_kernel(const float* part, int splits, const float* bias, const float2* rope,
                                                               __nv_bfloat16* qout, int n_q, int n_kv, int hd, __nv_bfloat16* kcache,
                                                               __nv_bfloat16* vcache, size_t layer_off, int max_seq, int L) {
    const int r = blockIdx.x, h2 = hd / 2, per_head = h2 / 4, n_qkv = (n_q + 2 * n_kv) * hd;
    const size_t stride = (size_t)gridDim.x * n_qkv;
    grid_dep_launch();
    grid_dep_wait();
    for (int it = threadIdx.x; it < (n_q + 2 * n_kv) * per_head; it += blockDim.x) {
        const int head = it / per_head, i = (it % per_head) * 4;
        const float* p = part + (size_t)r * n_qkv + head * hd + i;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (bias) {
            a = __ldg(reinterpret_cast<const float4*>(bias + head * hd + i));
            b = __ldg(reinterpret_cast<const float4*>(bias + head * hd + i + h2));
        }
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
            const float4* cs = reinterpret_cast<const float4*>(rope + (size_t)(L + r) * h2 + i);
            const float4 c0 = __ldg(cs), c1 = __ldg(cs + 1);
            lo = make_float4(a.x * c0.x - b.x * c0.y, a.y * c0.z - b.y * c0.w, a.z * c1.x - b.z * c1.y, a.w * c1.z - b.w * c1.w);
            hi = make_float4(b.x * c0.x + a.x * c0.y, b.y * c0.z + a.y * c0.w, b.z * c1.x + a.z * c1.y, b.w * c1.z + a.w * c1.w);
        }
        *reinterpret_cast<uint2*>(dst + i) = make_uint2(pack_bf16(lo.x, lo.y), pack_bf16(lo.z, lo.w));
        *reinterpret_cast<uint2*>(dst + i + h2) = make_uint2(pack_bf16(hi.x, hi.y), pack_bf16(hi.z, hi.w));
    }
}

// Causal attention of a sub-chunk's queries (rows r = 0..M-1 at positions L + r) over cache rows 0 .. L + r of their
// KV head.  A block holds the queries of all g heads that share a KV head: warp w takes the 16 queries of 16-row
// group w / g (of QT per block) and head w % g, so that a 64-key block fetched into shared memory (two cp.async
// buffers) serves g * QT warps.  The keys are cut into contiguous shares over the blocks of a cluster; every warp
// keeps scores, online softmax (log2 domain) and P V in registers (mma.sync m16n8k16), and the cluster's blocks
// merge their un-normalised outputs through distributed shared memory.  Output bf16 [M][n_q * hd].
// Bound by the mma.sync rate (a chunk's share of work per SM is 128 instructions per warp and 64 keys) and, over short
// contexts, by the chain load -> scores -> softmax -> merge.
template <int HD>
__global__ void __launch_bounds__(256) dense_attention_kernel(const __nv_bfloat16* q, const __nv_bfloat16* kcache,
                                                              const __nv_bfloat16* vcache, size_t layer_off, int max_seq, int n_q,
                                                              int g, int QT, int M, int L, float scale_log2e, __nv_bfloat16* out) {
    constexpr int KSTEPS = HD / 16, UNITS = HD / 8, NT_O = HD / 8, KB = 64;
    constexpr int KVBYTES = KB * HD * 2;
    extern __shared__ uint8_t att_smem_raw[];
    uint8_t* KVs = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(att_smem_raw) + 127) & ~(uintptr_t)127);   // [2 buffers][K | V]
    const int nthr = blockDim.x, nwarps = nthr >> 5;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
    const int CS = (int)cluster_size();
    const int rank = (int)cluster_rank();
    const int kvh = blockIdx.y, q0 = ((int)blockIdx.x / CS) * QT * 16;   // first query row of the block
    const int head = kvh * g + warp % g, r0 = q0 + (warp / g) * 16;      // this warp's head and first query row
    const size_t cache0 = layer_off + (size_t)kvh * max_seq * HD;
    const int nkeys = L + min(M, q0 + QT * 16);         // keys any row of this block may see
    const int nblk_all = (nkeys + KB - 1) / KB;
    const int b0 = even_start(nblk_all, CS, rank), nblk = even_count(nblk_all, CS, rank);
    auto load_block = [&](int blk) {
        if (blk < nblk) {
            uint8_t* Ks = KVs + (blk & 1) * 2 * KVBYTES;
            uint8_t* Vs = Ks + KVBYTES;
            for (int u = tid; u < KB * UNITS; u += nthr) {
                const int key = u / UNITS, q16 = u % UNITS, kk = (b0 + blk) * KB + key;
                const bool valid = kk < nkeys;
                const size_t off = cache0 + (size_t)(valid ? kk : 0) * HD + q16 * 8;
                const uint32_t so = (q16 >> 3) * (KB * 128) + swz_unit(key, q16 & 7);
                cp_async_16_zfill(Ks + so, kcache + off, valid);
                cp_async_16_zfill(Vs + so, vcache + off, valid);
            }
        }
        cp_async_commit();
    };
    grid_dep_launch();
    grid_dep_wait();
    load_block(0);
    load_block(1);
    const int gq = lane >> 2, q2 = (lane & 3) * 2;
    // query fragments stay in registers: rows gq and gq + 8 of the warp's 16, columns 16 ks + q2 (+ 8)
    uint32_t qf[KSTEPS][4];
    {
        const int rl = min(r0 + gq, M - 1), rh = min(r0 + gq + 8, M - 1);
        const uint32_t* pl = reinterpret_cast<const uint32_t*>(q + (size_t)rl * (n_q * HD) + head * HD + q2);
        const uint32_t* ph = reinterpret_cast<const uint32_t*>(q + (size_t)rh * (n_q * HD) + head * HD + q2);
#pragma unroll
        for (int ks = 0; ks < KSTEPS; ++ks) {
            qf[ks][0] = __ldcg(pl + ks * 8);
            qf[ks][1] = __ldcg(ph + ks * 8);
            qf[ks][2] = __ldcg(pl + ks * 8 + 4);
            qf[ks][3] = __ldcg(ph + ks * 8 + 4);
        }
    }
    float o[NT_O][4];
#pragma unroll
    for (int n = 0; n < NT_O; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
    float m_lo = -CUDART_INF_F, m_hi = -CUDART_INF_F, l_lo = 0.f, l_hi = 0.f;
    const int lim_lo = L + r0 + gq, lim_hi = lim_lo + 8;   // last key each row sees
    for (int blk = 0; blk < nblk; ++blk) {
        cp_async_wait<1>();
        __syncthreads();
        const uint32_t kb = smem_u32(KVs + (blk & 1) * 2 * KVBYTES), vb = kb + KVBYTES;
        const int key0 = (b0 + blk) * KB;
        if (key0 <= L + r0 + 15) {   // some key of this block is visible to some row of the warp
            float sc[KB / 8][4];
#pragma unroll
            for (int n = 0; n < KB / 8; ++n) sc[n][0] = sc[n][1] = sc[n][2] = sc[n][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < KSTEPS; ++ks) {
#pragma unroll
                for (int c = 0; c < KB / 16; ++c) {
                    uint32_t f0, f1, f2, f3;
                    const int krow = c * 16 + (lane & 7) + ((lane >> 4) << 3);
                    ldsm_x4(kb + (ks >> 2) * (KB * 128) + swz_unit(krow, (ks & 3) * 2 + ((lane >> 3) & 1)), f0, f1, f2, f3);
                    mma_bf16_16816(sc[2 * c], qf[ks][0], qf[ks][1], qf[ks][2], qf[ks][3], f0, f1);
                    mma_bf16_16816(sc[2 * c + 1], qf[ks][0], qf[ks][1], qf[ks][2], qf[ks][3], f2, f3);
                }
            }
            float mx_lo = -CUDART_INF_F, mx_hi = -CUDART_INF_F;
            const bool whole = key0 + KB - 1 <= L + r0;   // every key is visible to every row
#pragma unroll
            for (int n = 0; n < KB / 8; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int key = key0 + n * 8 + q2 + (e & 1);
                    const bool ok = whole || key <= (e >= 2 ? lim_hi : lim_lo);
                    const float v = ok ? sc[n][e] * scale_log2e : -CUDART_INF_F;
                    sc[n][e] = v;
                    if (e >= 2) mx_hi = fmaxf(mx_hi, v); else mx_lo = fmaxf(mx_lo, v);
                }
            mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 1));
            mx_lo = fmaxf(mx_lo, __shfl_xor_sync(0xffffffffu, mx_lo, 2));
            mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 1));
            mx_hi = fmaxf(mx_hi, __shfl_xor_sync(0xffffffffu, mx_hi, 2));
            const float mn_lo = fmaxf(m_lo, mx_lo), mn_hi = fmaxf(m_hi, mx_hi);
            const float use_lo = (mn_lo == -CUDART_INF_F) ? 0.f : mn_lo, use_hi = (mn_hi == -CUDART_INF_F) ? 0.f : mn_hi;
            const float c_lo = exp2f(m_lo - use_lo), c_hi = exp2f(m_hi - use_hi);
            m_lo = mn_lo;
            m_hi = mn_hi;
            float s_lo = 0.f, s_hi = 0.f;
            uint32_t pf[KB / 8][2];   // probabilities, packed: the A operand of the next product
#pragma unroll
            for (int n = 0; n < KB / 8; ++n) {
                const float p0 = exp2f(sc[n][0] - use_lo), p1 = exp2f(sc[n][1] - use_lo);
                const float p2 = exp2f(sc[n][2] - use_hi), p3 = exp2f(sc[n][3] - use_hi);
                s_lo += p0 + p1;
                s_hi += p2 + p3;
                pf[n][0] = pack_bf16(p0, p1);
                pf[n][1] = pack_bf16(p2, p3);
            }
            l_lo = l_lo * c_lo + s_lo;
            l_hi = l_hi * c_hi + s_hi;
#pragma unroll
            for (int n = 0; n < NT_O; ++n) { o[n][0] *= c_lo; o[n][1] *= c_lo; o[n][2] *= c_hi; o[n][3] *= c_hi; }
#pragma unroll
            for (int c = 0; c < KB / 16; ++c) {
#pragma unroll
                for (int cg = 0; cg < NT_O / 2; ++cg) {
                    uint32_t f0, f1, f2, f3;
                    const int key = c * 16 + (lane & 7) + (((lane >> 3) & 1) << 3);
                    const int cu = cg * 2 + (lane >> 4);
                    ldsm_x4_trans(vb + (cu >> 3) * (KB * 128) + swz_unit(key, cu & 7), f0, f1, f2, f3);
                    mma_bf16_16816(o[2 * cg], pf[2 * c][0], pf[2 * c][1], pf[2 * c + 1][0], pf[2 * c + 1][1], f0, f1);
                    mma_bf16_16816(o[2 * cg + 1], pf[2 * c][0], pf[2 * c][1], pf[2 * c + 1][0], pf[2 * c + 1][1], f2, f3);
                }
            }
        }
        __syncthreads();
        load_block(blk + 2);
    }
    cp_async_wait<0>();
    l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 1);
    l_lo += __shfl_xor_sync(0xffffffffu, l_lo, 2);
    l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 1);
    l_hi += __shfl_xor_sync(0xffffffffu, l_hi, 2);
    if (CS == 1) {
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int r = r0 + gq + half * 8;
            if (r >= M) continue;
            const float inv = 1.f / (half ? l_hi : l_lo);
            __nv_bfloat16* po = out + (size_t)r * (n_q * HD) + head * HD + q2;
#pragma unroll
            for (int n = 0; n < NT_O; ++n)
                *reinterpret_cast<uint32_t*>(po + n * 8) = pack_bf16(o[n][half * 2] * inv, o[n][half * 2 + 1] * inv);
        }
        return;
    }
    // the key shares meet: every block leaves its rows' outputs and statistics in its own shared memory (the K/V
    // buffers are free now) and then merges its share of the rows from all blocks of the cluster
    const int R = nwarps * 16;
    constexpr int LDO = HD + 4;
    float* ex_o = reinterpret_cast<float*>(KVs);            // [R][LDO]
    float2* ex_ml = reinterpret_cast<float2*>(ex_o + 128 * LDO);   // [R] (at most 128 rows)
    __syncthreads();
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const int lr = warp * 16 + gq + half * 8;
#pragma unroll
        for (int n = 0; n < NT_O; ++n)
            *reinterpret_cast<float2*>(ex_o + lr * LDO + n * 8 + q2) = make_float2(o[n][half * 2], o[n][half * 2 + 1]);
        if ((lane & 3) == 0) ex_ml[lr] = make_float2(half ? m_hi : m_lo, half ? l_hi : l_lo);
    }
    cluster_sync();
    {
        const uint32_t base_o = smem_u32(ex_o), base_ml = smem_u32(ex_ml);
        constexpr int C8 = HD / 8;
        const int rows_per = (R + CS - 1) / CS, rbeg = rank * rows_per, rend = min(R, rbeg + rows_per);
        for (int it = tid; it < (rend - rbeg) * C8; it += nthr) {
            const int lr = rbeg + it / C8, c = (it % C8) * 8;
            const int w = lr >> 4, r = q0 + (w / g) * 16 + (lr & 15);
            float2 ml[8];
            float mmax = -CUDART_INF_F;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k < CS) {
                    ml[k] = ld_cluster_f2(map_shared_rank(base_ml + lr * 8, k));
                    mmax = fmaxf(mmax, ml[k].x);
                }
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            float sum = 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k < CS) {
                    const uint32_t src = map_shared_rank(base_o + (lr * LDO + c) * 4, k);
                    const float4 x = ld_cluster_f4(src), y = ld_cluster_f4(src + 16);
                    const float wt = exp2f(ml[k].x - mmax);
                    sum += wt * ml[k].y;
                    a.x += wt * x.x; a.y += wt * x.y; a.z += wt * x.z; a.w += wt * x.w;
                    b.x += wt * y.x; b.y += wt * y.y; b.z += wt * y.z; b.w += wt * y.w;
                }
            if (r < M) {
                const float inv = 1.f / sum;
                *reinterpret_cast<uint4*>(out + (size_t)r * (n_q * HD) + (kvh * g + w % g) * HD + c) =
                    make_uint4(pack_bf16(a.x * inv, a.y * inv), pack_bf16(a.z * inv, a.w * inv), pack_bf16(b.x * inv, b.y * inv),
                               pack_bf16(b.z * inv, b.w * inv));
            }
        }
    }
    cluster_sync();   // no block leaves while another still reads its shared memory
}
template <int HD>
constexpr int dense_attention_smem() {
    constexpr int kv = 4 * 64 * HD * 2, ex = 128 * (HD + 4) * 4 + 128 * 8;
    return (kv > ex ? kv : ex) + 128;
}

// Calibration, "Sample": the b best ids of every row from the tiles' best kDenseTopMax (largest first, lowest id among
// equals).  One block per row.
__global__ void __launch_bounds__(256) dense_top_merge_kernel(DenseTopOut top, int ntiles, int b, int* succ /* [rows][b] */) {
    __shared__ float bv_s[8];
    __shared__ int bi_s[8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n = ntiles * kDenseTopMax;
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
