// The persistent forward kernel: one launch runs the decoder over M <= 32 token rows
// (a verify step over [T, x_1..x_k], or one tile of a prefill chunk).
//
// One thread block per SM, 12 warps:
//   warp 11      weight streamer: walks the block's static share of every GEMM in launch order
//                and keeps a ring of 32 KB shared-memory stages full with bulk asynchronous copies.
//                It never waits for activations or grid barriers, only for free ring slots, so HBM
//                traffic continues across operation boundaries.
//   warp 10      one thread issues the tensor-core instructions (tcgen05.mma, M = 128 weight
//                rows x N = 16 or 32 token rows x K = 16 per instruction): the streamed stage is the A
//                operand, the token rows, resident in shared memory for the whole operation, the
//                B operand; accumulators live in tensor memory (four buffers, so the next passes run while one
//                is read out).  A share of few weight rows (q|k|v) stacks slices of its K as rows.
//   warps 0..7   read the accumulators back (tcgen05.ld) and run the fused epilogues: warps 0..3 the
//                first accumulator of a pass, warps 4..7 the second (or, for passes of up to 128
//                rows, alternate pairs of token columns of the one accumulator).  The q|k|v epilogue finishes its
//                rows: slices, norm, bias, rotary embedding, cache append.
//   warps 0..9   build the token operand at the start of an operation (normalised rows, merge of the
//                split-KV partial results, ...) and meet the other blocks; warps 0..7 are the softmax of the attention
//                step, whose products (scores and outputs, keys on the M side) warp 9 issues.
// Code counts like data here: a layer's phases are 100 KB and more of instructions that every warp goes through once, so what is
// written out twice is fetched twice.  What a phase is prepared with, its operand build and the barrier are therefore
// written once per phase, and the stand-alone GEMM is a kernel of its own.
// A layer is four operations separated by a bounded grid barrier: QKV projection; attention;
// output projection (+ residual); gate|up with SwiGLU followed, inside the same block (or the two blocks of a cluster, which exchange
// their SwiGLU columns and take half of the rows each) and without a barrier, by the slice of the down projection (+ residual) that
// consumes these SwiGLU columns.
#pragma once
#include <math_constants.h>

#include "layout.cuh"
#include "ptx.cuh"

namespace sdv {

enum PhaseKind { PH_EMBED = 0, PH_QKV, PH_ATTN, PH_O, PH_GUD, PH_LM, PH_RAW };
constexpr int kPhasesPerLayer = 4;

// Phase numbering of a launch: 0 = embedding; 1 + 4*layer + {0..3} = QKV, attention, output
// projection, gate|up + down; 1 + 4*n_layers = LM head; 2 + 4*n_layers = stand-alone GEMM.
__host__ __device__ __forceinline__ int decode_phase(int ph, int n_layers, int& layer) {
    layer = 0;
    if (ph == 0) return PH_EMBED;
    if (ph == 1 + kPhasesPerLayer * n_layers) return PH_LM;
    if (ph == 2 + kPhasesPerLayer * n_layers) return PH_RAW;
    layer = (ph - 1) / kPhasesPerLayer;
    return PH_QKV + (ph - 1) % kPhasesPerLayer;
}
// The one or two streamed operations of a phase, in streaming order.
__device__ __forceinline__ int phase_ops(int kind, int (&ops)[2]) {
    switch (kind) {
        case PH_QKV: ops[0] = OP_QKV; return 1;
        case PH_O: ops[0] = OP_O; return 1;
        case PH_GUD: ops[0] = OP_GU; ops[1] = OP_DOWN; return 2;
        case PH_LM: ops[0] = OP_LM; return 1;
        case PH_RAW: ops[0] = OP_RAW; return 1;
        default: return 0;
    }
}
__device__ __forceinline__ const uint8_t* op_weights(const FwdParams& P, int op, int layer) {
    if (op == OP_LM) return P.wlm + P.op[OP_LM].w_off;
    if (op == OP_RAW) return P.wraw + P.op[OP_RAW].w_off;
    return P.wlayers + (unsigned long long)layer * P.layer_stride + P.op[op].w_off;
}

struct NormShape {
    int segs, seg_inv;   // segments per row; quotients by it are products with seg_inv, shifted by 16
    int per4, row_step;  // float4 columns per segment; warps that share a segment
    int group, adj;      // 16-byte units per column group of the operand; step to the next K slice beyond the columns'
    uint32_t inv;        // see norm_shape
};
struct MmaShape {
    uint32_t idesc, blo, bstep;            // instruction descriptor; token operand's descriptor and its column step
    int steps, last_steps;                 // column steps of a stage, and of the last one
};
struct Misc {
    uint64_t full[kMaxStages], empty[kMaxStages];
    uint64_t tmem_full[kAccBufs], tmem_empty[kAccBufs];
    uint64_t op_ready;    // the token operand of this block's next operation is complete (one arrival per builder warp)
    uint64_t act_ready;   // the SwiGLU operand of this block is complete (one arrival per epilogue warp, and the other block's bytes)
    uint64_t att_bar;     // a product of the attention step has completed
    uint64_t done_bar;    // last tensor-core instruction of the launch has completed
    uint32_t tmem_base;
    unsigned long long* prof_ptr;  // this block's profile words of the running phase (or null)
    int abort_flag;
    int skip;  // block-uniform copy of abort_flag, refreshed inside every grid barrier
    float sumsq[2][kMaxRows];  // sums of squares of the residual rows (this block's operand columns), of this phase and the one before
    float att_red[kEpilogueWarps][32];  // maxima and sums of a warp's keys, one query row per lane (attention step)
    Part part[OP_COUNT];  // this block's share of every operation
    NormShape shape[OP_COUNT];
    MmaShape mma[OP_COUNT];
    FwdParams P;          // block-local copy of the launch parameters
    // behind an abandoned wait, blocks of a pair only (leave_pair):
    int pair_passes;      // accumulator passes this block, which gave up, has gone through
    int pair_abort;       // the other one gave up; it writes this, and the next two: phases it has sent its columns in, plus one; it has all of ours
    int pair_theirs, pair_done;
};
static_assert(sizeof(Misc) <= kMiscSmemBytes, "misc shared memory");

// ------------------------------------------------------------------------------------------
// Grid barrier: every block adds one to a counter (release) and waits (bounded, acquire) until all have.  Called by all worker
// threads.  The last worker warp (which has the least of the phases' work) meets the other blocks; the others only announce
// themselves and work out what the next phase needs (`prepare`) meanwhile.  Returns, identically for all of them,
// whether some bounded wait in this block has been abandoned (the remaining phases then do no work).
constexpr int kBarrierWarp = kWorkerWarps - 1;
template <typename F>
__device__ __forceinline__ bool grid_barrier(const FwdParams& P, unsigned target, Misc* misc, int wtid, F prepare) {
    const bool meets = (wtid >> 5) == kBarrierWarp;
    if (!meets) named_bar_arrive(1, kWorkerThreads);
    prepare();
    if (meets) {
        named_bar_sync(1, kWorkerThreads);
        if ((wtid & 31) == 0) {
            red_release_add_u32(P.bar, 1u);  // no return value to wait for: polling starts at once
            uint64_t t0 = 0;  // the global timer is slow to read: only once the wait has lasted a while
            uint32_t spins = 0;
            while ((int)(ld_acquire_gpu_u32(P.bar) - target) < 0) {  // wrap-safe: the difference, read as signed
                if ((++spins & 63u) == 0) {
                    if (*(volatile int*)&misc->abort_flag) break;
                    const uint64_t now = global_timer_ns();
                    if (t0 == 0) t0 = now;
                    if (now - t0 > P.wait_limit_ns) {
                        *(volatile int*)&misc->abort_flag = 1;
                        break;
                    }
                }
            }
            *(volatile int*)&misc->skip = *(volatile int*)&misc->abort_flag;
        }
    }
    named_bar_sync(4, kWorkerThreads);
    return *(volatile int*)&misc->skip != 0;
}

// ------------------------------------------------------------------------------------------
// Weight streamer (one thread).  The ring holds 128 KB of the 590 KB a layer of the 1.5B shape streams per block, and HBM
// would idle through the attention half of a layer (24 us) once it is full.  So while the streamer waits for a free slot it reads
// ahead into L2, at most kLookaheadBytes beyond the ring and no faster than one piece per kLookaheadCycles or kLookaheadSlow
// (4 or 3 TB/s over the grid if nothing else ran): a burst would queue in front of the other warps' loads, which cost more than it gave, the trickle does not.
// Forward kernel without reading ahead, with 128, 256 and 384 KB: 1.5B shape, 9 rows, 2048 keys 956, 925, 905 and 904 us; 12 layers of the 7B
// shape, 5 rows, 8192 keys 1226, 1216, 1212 and 1209.
// The rate, by the time of the forward kernel at 800 cycles over that at 600 (by turns in one process, at 2048 | 8192 keys; a share is what a block
// streams of a layer, MB of 2^20 bytes):
//   1.5B shape (0.6 MB): 1, 5, 9 and 13 rows 1.013 1.018 1.016 1.018 | 1.008 1.007 0.988 0.990, 17 and 24 rows 1.000 1.002 | 0.981 1.026;
//     25 and 32 rows, where the operand builds are what a layer waits for, 0.999 0.992 | 1.007 1.015.
//   3B shape (1.3 MB): 1, 9, 17 and 24 rows 1.010 0.999 1.010 1.013 | 1.000 0.984 0.992 1.004; 25 rows 1.012 | 1.007.
//   2.2 MB: 1, 5 and 9 rows 1.007 1.009 1.016 | 1.010 1.011 1.009.  2.5 MB: 1.007 0.999 1.004 | 1.004 1.007 1.002.
//   7B shape (3.0 MB): 1, 5, 9 and 17 rows 1.009 1.008 1.006 1.015 | 1.002 0.998 1.001 1.002, at 256 keys 1.009 1.008 1.008 1.006.
// The two lines were drawn where layers took longer and the slow rate won by 0.3 to 1.2 % on their far sides.  Now it does so at 25 and 32 rows of the
// 1.5B shape up to 2048 keys, and costs up to 1.5 % elsewhere beyond them.  1100 cycles: 1.5B shape, 32 rows 0.978 | 0.969 and 25 rows 0.999 | 0.975
// of the time at 600, 1.02 times at up to 13 rows and 2048 keys; 7B shape 1.000 to 1.016 times.
struct Lookahead {   // cursor over the block's weight stream: operation by operation, each one contiguous range of bytes
    int ph, oi;
    const uint8_t* src;
    unsigned long long begin, end;   // the running operation's place in the stream
    uint32_t bytes, first;           // its bytes, and where in its weights the block begins
};
__device__ __forceinline__ bool lookahead_next(const FwdParams& P, Misc* misc, Lookahead& c) {
    for (;;) {
        int layer, ops[2];
        if (c.ph >= P.ph_end) return false;
        const int nops = phase_ops(decode_phase(c.ph, P.n_layers, layer), ops);
        if (++c.oi >= nops) { c.oi = -1; ++c.ph; continue; }
        const Part& pt = misc->part[ops[c.oi]];
        if (pt.ntiles == 0 || pt.nk == 0) continue;
        c.src = op_weights(P, ops[c.oi], layer) + pt.off;
        c.begin = c.end;
        c.bytes = (uint32_t)(pt.ntiles * pt.nk * kStepBytes);
        c.first = (uint32_t)(pass_start(pt, pt.rot) * pt.nk * kStepBytes);
        c.end += c.bytes;
        return true;
    }
}
__device__ __forceinline__ void producer_loop(const FwdParams& P, uint8_t* smem, Misc* misc) {
    const uint64_t policy = l2_policy_evict_first();
    const uint32_t nstage = (uint32_t)P.nstage;
    uint32_t slot = 0, par = 0, issued = 0;  // ring position; parity of the current trip round the ring
    bool ok = true;
    unsigned long long streamed = 0, ahead = 0;   // bytes copied / read ahead so far
    Lookahead la;
    la.ph = P.ph_begin; la.oi = -1; la.begin = la.end = 0; la.src = nullptr; la.bytes = la.first = 0;
    bool more = lookahead_next(P, misc, la);
    const uint32_t pause = P.M > kLookaheadRows || P.layer_stride > kLookaheadShare * (unsigned)P.G ? kLookaheadSlow : kLookaheadCycles;
    uint32_t last = (uint32_t)clock64();
#pragma unroll 1
    for (int ph = P.ph_begin; ph < P.ph_end && ok; ++ph) {
        int layer, ops[2];
        const int kind = decode_phase(ph, P.n_layers, layer);
        const int nops = phase_ops(kind, ops);
#pragma unroll 1
        for (int oi = 0; oi < nops && ok; ++oi) {
            const Part& pt = misc->part[ops[oi]];
            if (pt.ntiles == 0 || pt.nk == 0) continue;
            const uint8_t* const op_src = op_weights(P, ops[oi], layer) + pt.off;
            const int nst = pt.nst, SK = pt.SK, nk = pt.per;
#pragma unroll 1
            for (int p = 0; p < pt.npass && ok; ++p) {
                const int pi = pass_index(pt, p);
                const uint8_t* src = op_src + (size_t)pass_start(pt, pi) * (uint32_t)(pt.nk * kStepBytes);
                const uint32_t pbytes = (uint32_t)(pass_count(pt, pi) * pt.slices) * kStepBytes;
                int kleft = nk;
#pragma unroll 1
                for (int st = 0; st < nst; ++st, kleft -= SK) {
                    const uint32_t bytes = pbytes * (uint32_t)min(SK, kleft);
                    // the slot's previous contents must have been consumed (first trip: free at once)
                    uint64_t t0 = 0;
                    uint32_t spins = 0;
                    while (!mbar_test(&misc->empty[slot], par ^ 1u)) {
                        const uint32_t now = (uint32_t)clock64();
                        if (now - last > pause && more) {
                            if (ahead < streamed) ahead = streamed;
                            while (more && ahead >= la.end) more = lookahead_next(P, misc, la);
                            if (more && ahead < streamed + kLookaheadBytes) {
                                uint32_t at = (uint32_t)(ahead - la.begin) + la.first, left = (uint32_t)(la.end - ahead);
                                if (at >= la.bytes) at -= la.bytes;
                                if (left > la.bytes - at) left = la.bytes - at;
                                const uint32_t piece = left < kLookaheadPiece ? left : kLookaheadPiece;
                                bulk_prefetch_l2(la.src + at, piece);
                                ahead += piece;
                                last = now;
                            }
                        }
                        if ((++spins & 255u) == 0) {
                            if (*(volatile int*)&misc->abort_flag) { ok = false; break; }
                            const uint64_t t = global_timer_ns();
                            if (t0 == 0) t0 = t;
                            if (t - t0 > P.wait_limit_ns) { *(volatile int*)&misc->abort_flag = 1; ok = false; break; }
                        }
                    }
                    if (!ok) break;
                    mbar_arrive_expect_tx(&misc->full[slot], bytes);
                    bulk_g2s(smem + slot * kStageBytes, src, bytes, &misc->full[slot], policy);
                    src += bytes;
                    streamed += bytes;
                    ++issued;
                    if (++slot == nstage) { slot = 0; par ^= 1u; }
                }
            }
        }
    }
    // The copies still in flight are waited for (bounded) before the block may exit: where a wait was given up, here or later, nobody else does.
    for (uint32_t back = 0; back < nstage && back < issued; ++back) {
        if (slot == 0) { slot = nstage; par ^= 1u; }
        --slot;
        if (!mbar_drain(&misc->full[slot], par, P.wait_limit_ns)) break;
    }
}

// ------------------------------------------------------------------------------------------
// Token operand of a GEMM, resident in shared memory for the whole operation, in a layout the
// tensor core reads (K-major, no swizzle): for every 8 columns the M token rows, 16 bytes each:
//     [8-column group][row 0..M-1, padded to an odd number where it fits][8 bf16].
// An 8-row core matrix is 128 contiguous bytes, row groups are 128 bytes apart and the two halves
// of a column step M * 16 bytes.  The instruction reads 16 or 32 rows: the ones past M belong to the
// next column groups (or lie behind the operand, still inside shared memory) and only feed
// accumulator columns nobody reads.
__device__ __forceinline__ uint32_t operand_off(int k8, int row, int M) {  // M: operand_rows()
    return (uint32_t)((k8 * M + row) * 16);
}

// Operand = residual rows scaled by the RMSNorm weight (the per-row factor rsqrt(mean + eps)
// commutes with the GEMM and is applied by the consumer of the result), or, for the stand-alone
// GEMM, the caller's fp32 rows as they are.  The columns are cut into segments of up to kSegUnits units (32 lanes x 4 columns); a
// warp stays with one segment and takes every row_step-th row, loading the next row while it converts the one before.  So the
// norm weights and the places its columns go to are fixed: both are fetched or worked out while the blocks meet at
// the grid barrier before the phase (NormPrep), and a row costs 15 instructions per unit.  (With weights and addresses
// worked out per row and unit the build took 8 us at 32 rows of 1536 columns, 6 of them without loading a single row.)
// Leaves the rows' sums of squares over this block's columns in misc->sumsq.
constexpr int kSegUnits = 8;
struct NormPrep {
    const float4* src;       // first row of this warp, this lane's first column
    int step4;               // float4 columns from one of its rows to the next
    int row0, row_step;      // its rows
    int rem;                 // float4 columns from the lane's first one to the segment's end
    float4 w[kSegUnits];     // norm weights
    uint32_t off[kSegUnits]; // where a unit goes for row 0, bytes from the operand's start
};
// How the block's share of an operation is cut: the same in every layer, so its divisions are done once per launch.
__device__ __forceinline__ NormShape norm_shape(const FwdParams& P, const Part& pt) {
    NormShape f;
    const int units = (pt.nk * 4 + 31) >> 5;
    f.segs = max(1, (units + kSegUnits - 1) / kSegUnits);
    f.seg_inv = 65536 / f.segs + 1;
    f.per4 = (units + f.segs - 1) / f.segs * 32;
    f.row_step = max(1, kBuilderWarps / f.segs);
    f.group = operand_rows(P, P.M, pt.slices);
    const int slice4 = pt.nk * 4 / pt.slices;                               // float4 columns per slice (a multiple of 4)
    f.inv = pt.slices > 1 && slice4 > 0 ? 0xffffffffu / (uint32_t)slice4 + 1u : 0u;   // slice of a column = upper half of its product with inv
    f.adj = P.M - (slice4 >> 1) * f.group;                                  // step from a slice to the next beyond the columns'
    return f;
}
// `more` > 0: the warp's further segments, where a row has more of them than there are warps.
template <int KIND>
__device__ __forceinline__ void norm_prep(NormPrep& n, const FwdParams& P, const Misc* misc, int layer, int wtid, int more) {
    constexpr bool raw = KIND == PH_RAW;
    constexpr int op = KIND == PH_QKV ? OP_QKV : KIND == PH_GUD ? OP_GU : KIND == PH_LM ? OP_LM : OP_RAW;
    const NormShape& f = misc->shape[op];
    const Part& pt = misc->part[op];
    const int warp = wtid >> 5, lane = wtid & 31;
    const int stride4 = (raw ? P.raw_K : P.d) >> 2, k4_0 = pt.k0 * 4, nk4 = pt.nk * 4;
    const int turn = (warp * f.seg_inv) >> 16, seg = warp - turn * f.segs + more;
    n.row_step = f.row_step;
    n.row0 = turn < f.row_step ? turn : kMaxRows;
    const int c0 = seg * f.per4 + lane;
    n.rem = min(f.per4, nk4 - seg * f.per4) - lane;
    n.src = reinterpret_cast<const float4*>(raw ? P.raw_x : P.h) + n.row0 * stride4 + k4_0 + c0;
    n.step4 = n.row_step * stride4;
    const float4* w = reinterpret_cast<const float4*>(P.norm_w + (size_t)(KIND == PH_QKV ? layer * 2 : KIND == PH_GUD ? layer * 2 + 1 : P.n_layers * 2) * P.d) + k4_0 + c0;
#pragma unroll
    for (int u = 0; u < kSegUnits; ++u) {
        n.w[u] = raw ? make_float4(1.f, 1.f, 1.f, 1.f) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (!raw) ld_nc_f4_gt(n.w[u], w + u * 32, n.rem, u * 32);
    }
#pragma unroll
    for (int u = 0; u < kSegUnits; ++u) {
        const int k4 = c0 + u * 32;
        n.off[u] = (uint32_t)(((k4 >> 1) * f.group + (int)__umulhi((uint32_t)k4, f.inv) * f.adj) * 16 + (k4 & 1) * 8);
    }
}
__device__ __forceinline__ void norm_load(const NormPrep& n, float4 (&a)[kSegUnits], const float4* src, bool live) {
    const int rem = live ? n.rem : 0;
#pragma unroll
    for (int u = 0; u < kSegUnits; ++u) ld_cg_f4_gt(a[u], src + u * 32, rem, u * 32);
}
__device__ __forceinline__ void norm_convert(const NormPrep& n, const float4 (&a)[kSegUnits], uint32_t dst, float* sumsq, bool one, int lane) {
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int u = 0; u < kSegUnits; ++u) {
        const float4 v = a[u], g = n.w[u];
        s0 += v.x * v.x + v.y * v.y;
        s1 += v.z * v.z + v.w * v.w;
        st_shared_v2_gt(dst + n.off[u], pack_bf16(v.x * g.x, v.y * g.y), pack_bf16(v.z * g.z, v.w * g.w), n.rem, u * 32);
    }
    s0 += s1;
#pragma unroll
    for (int off = 16; off; off >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, off);
    if (lane == 0) {
        if (one) *sumsq = s0;
        else atomicAdd(sumsq, s0);
    }
}
// `buf`: which of the two sets of sums this phase uses; the other one is cleared for the next.
template <int KIND>
__device__ __forceinline__ void build_norm_operand(const FwdParams& P, NormPrep& n, int layer, uint8_t* U, Misc* misc, int buf, int wtid) {
    constexpr int op = KIND == PH_QKV ? OP_QKV : KIND == PH_GUD ? OP_GU : KIND == PH_LM ? OP_LM : OP_RAW;
    const int lane = wtid & 31, M = P.M, segs = misc->shape[op].segs;
    float* sumsq = misc->sumsq[buf];
    if (wtid < kMaxRows) misc->sumsq[buf ^ 1][wtid] = 0.f;
    const uint32_t dst = smem_u32(U);
#pragma unroll 1
    for (int more = 0;;) {
        float4 a[kSegUnits], b[kSegUnits];
#pragma unroll
        for (int u = 0; u < kSegUnits; ++u) a[u] = b[u] = make_float4(0.f, 0.f, 0.f, 0.f);   // units past the segment stay zero
        const float4* src = n.src;
        int row = n.row0;
        norm_load(n, b, src, row < M);
#pragma unroll 1
        while (row < M) {
#pragma unroll
            for (int u = 0; u < kSegUnits; ++u) a[u] = b[u];
            src += n.step4;
            norm_load(n, b, src, row + n.row_step < M);
            norm_convert(n, a, dst + (uint32_t)row * 16u, sumsq + row, segs == 1, lane);
            row += n.row_step;
        }
        more += kBuilderWarps;
        if (segs <= kBuilderWarps || (wtid >> 5) + more >= segs) break;
        norm_prep<KIND>(n, P, misc, layer, wtid, more);
    }
}

// Operand of the output projection = attention output of this block's columns: the split-KV
// partial results (un-normalised sums with their running maximum and sum) are merged on the way.
// LPI lanes share one (row, 8 columns) item, each taking every LPI-th partial result, TPL of them at most.  A round of items waits for one trip
// to L2 (1.4 us, the loads of all its partial results in flight together), so the items should fit one round: four lanes an
// item up to kWorkerThreads / 4 items, two lanes above where the results are at most 20 (1.5B shape, 2048 keys: 21 rows 6.6 -> 5.7 us
// a phase, 32 rows 7.0 -> 6.4; at 9 rows, one round either way, four lanes are 0.1 to 0.3 us faster).
template <int LPI, int TPL>
__device__ __forceinline__ void build_merged_operand(const FwdParams& P, const Part& pt, uint8_t* U, int wtid) {
    const int S = P.att_S;
    const int M = P.M, Mp = operand_rows(P, P.M, 1), hd = P.hd;
    const int k8_0 = pt.k0 * 2, nk8 = pt.nk * 2;
    const int nitems = M * nk8, sub = wtid % LPI;
#pragma unroll 1
    for (int it0 = 0; it0 < nitems; it0 += kBuilderWarps * 32 / LPI) {
        const int item = it0 + wtid / LPI;
        const bool live = item < nitems;
        const int j = live ? item / nk8 : 0, k8l = live ? item % nk8 : 0;
        const int col = (k8_0 + k8l) * 8, hq = col / hd, c = col % hd;
        const size_t base = ((size_t)hq * kMaxSplits) * kMaxRows + j;
        float m[TPL], l[TPL];
        float4 a[TPL], b[TPL];
        // every slot loads (beyond the last partial result: the last one again, given no weight below), so that
        // the loads are one straight run of instructions instead of a branch per slot
#pragma unroll
        for (int t = 0; t < TPL; ++t) {
            const int s = sub + LPI * t;
            const size_t row = base + (size_t)min(s, S - 1) * kMaxRows;
            const float2 ml = ld_cg_f2_inorder(P.part_ml + row * 2);
            const float* op = P.part_o + row * hd + c;
            a[t] = ld_cg_f4_inorder(op);
            b[t] = ld_cg_f4_inorder(op + 4);
            const bool use = live && s < S;
            m[t] = use ? ml.x : -CUDART_INF_F;
            l[t] = use ? ml.y : 0.f;
        }
        float mmax = m[0];
#pragma unroll
        for (int t = 1; t < TPL; ++t) mmax = fmaxf(mmax, m[t]);
#pragma unroll
        for (int off = 1; off < LPI; off <<= 1) mmax = fmaxf(mmax, __shfl_xor_sync(0xffffffffu, mmax, off));
        const float ref = (mmax == -CUDART_INF_F) ? 0.f : mmax;
        float v[9];
#pragma unroll
        for (int e = 0; e < 9; ++e) v[e] = 0.f;
#pragma unroll
        for (int t = 0; t < TPL; ++t) {
            const float w = exp2f(m[t] - ref);  // 0 for partial results that saw no key
            v[0] += w * a[t].x; v[1] += w * a[t].y; v[2] += w * a[t].z; v[3] += w * a[t].w;
            v[4] += w * b[t].x; v[5] += w * b[t].y; v[6] += w * b[t].z; v[7] += w * b[t].w;
            v[8] += w * l[t];
        }
#pragma unroll
        for (int e = 0; e < 9; ++e) {
#pragma unroll
            for (int off = 1; off < LPI; off <<= 1) v[e] += __shfl_xor_sync(0xffffffffu, v[e], off);
        }
        if (live && sub == 0) {
            const float inv = 1.f / v[8];
            const uint4 out = make_uint4(pack_bf16(v[0] * inv, v[1] * inv), pack_bf16(v[2] * inv, v[3] * inv),
                                         pack_bf16(v[4] * inv, v[5] * inv), pack_bf16(v[6] * inv, v[7] * inv));
            *reinterpret_cast<uint4*>(U + operand_off(k8l, j, Mp)) = out;
        }
    }
}

// ------------------------------------------------------------------------------------------
// Tensor-core issue, by one thread for the whole launch.  Measured on the part: the pipe takes an instruction (M = 128, N <= 32) every
// 39 cycles and a commit costs it 87, so a 32 KB stage (eight instructions, a commit) takes 399; about eight entries wait in its queue.  The
// issuing thread pays the full latency of every dependent instruction and branch, so it keeps up only if nothing but the instructions stands
// between a commit and the next one: an operation is one flat loop over its (pass, stage) pairs, what the next pair needs is worked
// out and its barriers are looked at (without waiting) behind this pair's instructions and before its commits, barriers go by
// their shared-memory addresses, and what is the same all through an operation is worked out once per launch (MmaShape).
// Stand-alone, with nothing to wait for, in cycles (before: nested loops, commits first): gate|up of the 0.5B shape 5595 -> 3971, the 1.5B
// shape 8569 -> 5945; down 7584 -> 4069, 3B shape 14257 -> 6945; output projection 2826 -> 1717; a 16-tile share over 160 column steps
// 26054 -> 16473.
// Pipeline positions: (slot, par) is the ring position (slot index and parity of the current trip round the ring), `q`
// counts accumulator passes, `ops` token operands; all advance over the whole launch, identically in every role.
struct PipePos {
    uint32_t slot, par, q, ops, sums;
    uint32_t w_full, w_acc;  // cycles the tensor-core thread waited for weights / for a free accumulator (profile)
};
__device__ __forceinline__ MmaShape mma_shape(const FwdParams& P, const Part& pt, uint32_t operand) {
    MmaShape f;
    const int brows = pt.slices * P.M;                          // rows of the token operand (stacked K slices)
    const uint32_t lbo_b = (uint32_t)operand_rows(P, P.M, pt.slices) * 16u;
    f.idesc = umma_idesc_bf16_m128(pt.slices > 1 ? (uint32_t)((brows + 15) & ~15) : (uint32_t)P.NB);
    f.blo = umma_smem_lo(operand, lbo_b);
    f.bstep = (2u * lbo_b) >> 4;                                // one column step, in descriptor address units
    f.steps = pt.SK;
    f.last_steps = pt.per - (pt.nst - 1) * pt.SK;
    return f;
}

// Barriers by their shared-memory addresses.
__device__ __forceinline__ bool mbar_test_at(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void umma_commit_at(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// One operation; one or (TWO) two 128-row accumulators per pass (where some passes of an operation need the second one, all are given it: its
// instructions read on behind a shorter pass's rows, inside shared memory, into columns nobody reads; only shares of 17 tiles, passes of nine and
// eight, issue more for it).  The token operand is waited
// for last, with everything else at hand.  due_slot, due_acc: commits that are due behind the last instructions issued.  False: a
// wait was abandoned.
template <bool TWO>
__device__ __forceinline__ bool mma_stages(const FwdParams& P, const Part& pt, const MmaShape& fs, uint32_t ring0, Misc* misc, PipePos& pos, bool& ready, uint64_t* operand,
                                           uint32_t operand_par) {
    constexpr int GROUP = TWO ? 4 : 8;
    const uint32_t bstep = fs.bstep, idesc = fs.idesc, blo = fs.blo, nstage = (uint32_t)P.nstage;
    const int steps = fs.steps, last_steps = fs.last_steps, nst = pt.nst;
    const uint64_t wait_limit = P.wait_limit_ns;
    const uint32_t full0 = smem_u32(&misc->full[0]), empty0 = smem_u32(&misc->empty[0]), acc_full0 = smem_u32(&misc->tmem_full[0]), acc_empty0 = smem_u32(&misc->tmem_empty[0]);
    const uint32_t tmem0 = misc->tmem_base, dstep = pt.slices > 1 ? 0u : kTmemBuf, dbase = tmem0 + (pt.slices > 1 ? kTmemStack : 0u);
    const int prem = pt.prem;
    uint32_t buf = pos.q % kAccBufs, apar = ((pos.q / kAccBufs) & 1u) ^ 1u, slot = pos.slot, par = pos.par;
    int pi = pt.rot, p = pt.npass, st = nst;
    uint32_t count = (uint32_t)((pt.pbase + (pi < prem ? 1 : 0)) * pt.slices), alo = umma_smem_lo(ring0, count * 256u), astep = count * 32u;
    uint32_t d = dbase + buf * dstep, b = blo, acc = 0u, due_slot = 0u, due_acc = 0u;
    if (!mbar_test_at(acc_empty0 + buf * 8u, apar)) {
        const long long t0 = clock64();
        if (!mbar_wait_bounded(&misc->tmem_empty[buf], apar, &misc->abort_flag, wait_limit)) return false;
        pos.w_acc += (uint32_t)(clock64() - t0);
    }
    if (!ready) {
        const long long t0 = clock64();
        if (!mbar_wait_bounded(&misc->full[slot], par, &misc->abort_flag, wait_limit)) return false;
        pos.w_full += (uint32_t)(clock64() - t0);
    }
    if (!mbar_wait_bounded(operand, operand_par, &misc->abort_flag, wait_limit)) return false;
#pragma unroll 1
    for (;;) {
        tc_fence_after();
        if (due_slot) umma_commit_at(due_slot);
        if (due_acc) umma_commit_at(due_acc);
        due_acc = 0u;
        uint32_t a = alo + slot * (uint32_t)(kStageBytes >> 4);
        int left = st == 1 ? last_steps : steps;
        if (left == GROUP) {
#pragma unroll
            for (int i = 0; i < GROUP; ++i) {
                umma_bf16_lo(d, a + i * astep, b + i * bstep, idesc, i == 0 ? acc : 1u);
                if (TWO) umma_bf16_lo(d + 32u, a + i * astep + 128u, b + i * bstep, idesc, i == 0 ? acc : 1u);   // rows 128.. of the pass
            }
            b += GROUP * bstep;
        } else {
#pragma unroll 1
            for (; left > 1; left -= 2) {
                umma_bf16_lo(d, a, b, idesc, acc);
                if (TWO) umma_bf16_lo(d + 32u, a + 128u, b, idesc, acc);
                umma_bf16_lo(d, a + astep, b + bstep, idesc, 1u);
                if (TWO) umma_bf16_lo(d + 32u, a + astep + 128u, b + bstep, idesc, 1u);
                acc = 1u;
                a += 2u * astep;
                b += 2u * bstep;
            }
            if (left > 0) {
                umma_bf16_lo(d, a, b, idesc, acc);
                if (TWO) umma_bf16_lo(d + 32u, a + 128u, b, idesc, acc);
                b += bstep;
            }
        }
        acc = 1u;
        due_slot = empty0 + slot * 8u;
        if (++slot == nstage) { slot = 0; par ^= 1u; }
        ready = mbar_test_at(full0 + slot * 8u, par);   // the next stage, of this operation or the one after
        if (--st == 0) {
            due_acc = acc_full0 + buf * 8u;
            buf = (buf + 1u) % kAccBufs;
            if (buf == 0u) apar ^= 1u;
            if (--p == 0) break;
            st = nst;
            b = blo;
            acc = 0u;
            d = dbase + buf * dstep;
            if (prem) {
                if (++pi == pt.npass) pi = 0;
                count = (uint32_t)((pt.pbase + (pi < prem ? 1 : 0)) * pt.slices);
                alo = umma_smem_lo(ring0, count * 256u);
                astep = count * 32u;
            }
            if (!mbar_test_at(acc_empty0 + buf * 8u, apar)) {
                umma_commit_at(due_slot);
                umma_commit_at(due_acc);
                due_slot = due_acc = 0u;
                const long long t0 = clock64();
                if (!mbar_wait_bounded(&misc->tmem_empty[buf], apar, &misc->abort_flag, wait_limit)) return false;
                pos.w_acc += (uint32_t)(clock64() - t0);
            }
        }
        if (!ready) {
            if (due_slot) umma_commit_at(due_slot);
            if (due_acc) umma_commit_at(due_acc);
            due_slot = due_acc = 0u;
            const long long t0 = clock64();
            if (!mbar_wait_bounded(&misc->full[slot], par, &misc->abort_flag, wait_limit)) return false;
            pos.w_full += (uint32_t)(clock64() - t0);
        }
    }
    umma_commit_at(due_slot);
    umma_commit_at(due_acc);
    pos.slot = slot;
    pos.par = par;
    pos.q += (uint32_t)pt.npass;
    return true;
}
__device__ __forceinline__ bool mma_op(const FwdParams& P, int op, uint32_t ring0, Misc* misc, PipePos& pos, bool& ready, uint64_t* operand,
                                       uint32_t operand_par) {
    const Part& pt = misc->part[op];
    const MmaShape f = misc->mma[op];
    return (pt.pbase + (pt.prem > 0 ? 1 : 0)) * pt.slices > 8 ? mma_stages<true>(P, pt, f, ring0, misc, pos, ready, operand, operand_par)
                                                              : mma_stages<false>(P, pt, f, ring0, misc, pos, ready, operand, operand_par);
}

// ------------------------------------------------------------------------------------------
// Epilogues (warps 0..7).  Thread t = 32 * (warp & 3) + lane owns row t of its 128-row accumulator,
// i.e. one weight row (output feature), for the token columns its warp group takes.  Token columns are taken 16 at a time.
// SwiGLU on one accumulator row per thread.  Rows 0..7 of a 16-row tile are gate rows, rows 8..15 the
// matching up rows, so the two values of an output sit 8 lanes apart.  Token columns are taken in
// pairs: the gate lane evaluates the even column of a pair, the up lane the odd one; one shuffle per
// pair hands each lane the partner's value it needs.  All pairs are independent and written without
// branches, so that their shuffles, exponentials and divisions overlap.  SEL >= 0: only pairs j with
// (j & 1) == SEL (the other group of epilogue warps takes the rest).  rs: lane n holds the norm factor of token n;
// n0: first token column of v, M: token columns from there on.
template <int SEL>
__device__ __forceinline__ void swiglu_pairs(const float (&v)[16], float rs, int n0, int t, bool valid, int M, uint8_t* dst) {
    constexpr int STEP = SEL < 0 ? 1 : 2, J0 = SEL < 0 ? 0 : SEL, NP = (8 - J0 + STEP - 1) / STEP;
    const bool is_up = (t & 8) != 0;
    float got[NP], out[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        const int j = J0 + i * STEP;
        got[i] = __shfl_xor_sync(0xffffffffu, is_up ? v[2 * j] : v[2 * j + 1], 8);
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        const int j = J0 + i * STEP;
        const float mine = is_up ? v[2 * j + 1] : v[2 * j], r = __shfl_sync(0xffffffffu, rs, n0 + 2 * j + (is_up ? 1 : 0));
        const float x = (is_up ? got[i] : mine) * r, y = (is_up ? mine : got[i]) * r;
        out[i] = __fdividef(x, 1.f + __expf(-x)) * y;
    }
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        const int n = 2 * (J0 + i * STEP) + (is_up ? 1 : 0);
        if (valid && n < M) *reinterpret_cast<__nv_bfloat16*>(dst + n * 16) = __float2bfloat16(out[i]);
    }
}

// Running best logit of each token row (LM head), per thread.
struct Best {
    float v[2][16];
    int i[2][16];
};

// op: the operation; with the LM head `best` carries the running best logits.
template <int op>
__device__ __forceinline__ void epilogue_op(const FwdParams& P, const Part& pt, uint8_t* act, Misc* misc, PipePos& pos, bool& dead,
                                            int warp, int lane, Best& best) {
    constexpr bool LM = op == OP_LM;
    const int M = P.M, Mp = operand_rows(P, P.M, 1);
    const int quarter = warp & 3, myhalf = warp >> 2;  // this warp's 32 accumulator lanes; which of the two accumulators
    const int t = quarter * 32 + lane;
    const uint64_t wait_limit = P.wait_limit_ns;
    const uint32_t tmem_lane = misc->tmem_base + ((uint32_t)(quarter * 32) << 16);
    const int npass = pt.npass, tile0 = pt.tile0, nchunk = M > 16 ? 2 : 1;
    float rs = 0.f;   // lane n: norm factor of token n
    if ((op == OP_GU || LM) && lane < M) rs = rsqrtf(misc->sumsq[pos.sums][lane] * (1.f / (float)P.d) + P.eps);
    float* out = P.h;
    int stride = P.d;
    bool add = true;  // residual add (O, down)
    if (op == OP_RAW) { out = P.raw_out; stride = P.raw_N; add = P.op[OP_RAW].P_k > 1; }
    const int store_logits = P.store_logits;
    const Part& down = misc->part[OP_DOWN];
    const int act_col0 = op == OP_GU ? (pt.tile0 / 2 - down.k0) * 16 : 0;   // gate|up has two tiles to a column step of the down projection
#pragma unroll 1
    for (int p = 0; p < npass; ++p, ++pos.q) {
        const int pi = op == OP_GU || LM ? p : pass_index(pt, p);   // those two have no partial sums
        const int pcount = pass_count(pt, pi), pstart = pass_start(pt, pi);
        const uint32_t buf = pos.q % kAccBufs;
        if (!dead && !mbar_wait_bounded(&misc->tmem_full[buf], (pos.q / kAccBufs) & 1u, &misc->abort_flag, wait_limit)) dead = true;
        dead = __any_sync(0xffffffffu, dead);
        if (dead) continue;
        tc_fence_after();
        if (misc->prof_ptr && t == 0 && p == npass - 1) misc->prof_ptr[10] = global_timer_ns();
        const int nhalf = pcount > 8 ? 2 : 1;  // a pass of more than 8 tiles fills both 128-row accumulators of the buffer
        // two accumulators: warps 0..3 read the first, 4..7 the second; one accumulator: both groups read
        // it and share its token columns (pairs of columns alternate between the groups)
        const int nsel = (nhalf == 2) ? -1 : myhalf;
        const int half = (nhalf == 2) ? myhalf : 0;
        const uint32_t taddr = tmem_lane + buf * kTmemBuf + (uint32_t)half * 32u;
        const int tt = half * 128 + t;         // row within the pass
        const bool valid = tt < 16 * pcount;
        const int row = (tile0 + pstart) * 16 + tt;  // weight row = output feature
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h == 0 || nchunk == 2) {
                float v[16];
                tmem_ld16(taddr + (uint32_t)(h * 16), v);
                if (h + 1 == nchunk) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&misc->tmem_empty[buf]);  // this warp's part of the accumulators may be overwritten
                }
                const int n0 = h * 16, Mh = M - n0;
                if (LM) {
#pragma unroll
                    for (int n = 0; n < 16; ++n) {
                        const float r = __shfl_sync(0xffffffffu, rs, n0 + n);
                        if (valid && n < Mh && (nsel < 0 || ((n >> 1) & 1) == nsel)) {
                            const float x = v[n] * r;
                            if (store_logits) __stcg(P.logits + (size_t)(n0 + n) * P.V + row, x);
                            // rows come in ascending order per thread, so ">" keeps the lowest id among equals
                            if (x > best.v[h][n]) { best.v[h][n] = x; best.i[h][n] = row; }
                        }
                    }
                } else if (op == OP_GU) {
                    // rows 0..7 of a tile are gate rows, 8..15 the matching up rows, 8 lanes apart: the gate
                    // lane evaluates the even token columns, the up lane the odd ones
                    const int col = (pstart + (tt >> 4)) * 8 + (tt & 7) + act_col0;  // SwiGLU column within the down projection's share
                    uint8_t* dst = act + operand_off(col >> 3, n0, Mp) + (col & 7) * 2;
                    if (nsel < 0) swiglu_pairs<-1>(v, rs, n0, t, valid, Mh, dst);
                    else if (nsel == 0) swiglu_pairs<0>(v, rs, n0, t, valid, Mh, dst);
                    else swiglu_pairs<1>(v, rs, n0, t, valid, Mh, dst);
                } else if (valid) {
                    float* d2 = out + (size_t)n0 * stride + row;
                    if (add) {
#pragma unroll
                        for (int n = 0; n < 16; ++n, d2 += stride)
                            if (n < Mh && (nsel < 0 || ((n >> 1) & 1) == nsel)) red_add_f32(d2, v[n]);
                    } else {
#pragma unroll
                        for (int n = 0; n < 16; ++n, d2 += stride)
                            if (n < Mh && (nsel < 0 || ((n >> 1) & 1) == nsel)) __stcg(d2, v[n]);
                    }
                }
            }
        }
    }
    if (!LM && op == OP_GU) {
        // this warp's SwiGLU columns are written: hand them to the tensor-core thread; the blocks of a pair send each other theirs, which lie
        // one behind the other in the operand (one copy of some KB; both wait for it, so neither is ahead by more than this).  They are sent
        // behind an abandoned wait as well, so that the phases prepared for and the copies sent stay the same number (pair_debt).
        fence_proxy_async_smem();
        const int steps = pt.ntiles / 2, theirs = down.nk - steps;
        if (theirs > 0) {
            named_bar_sync(2, kEpilogueWarps * 32);
            if (warp == 0 && lane == 0) {
                const uint32_t peer = cluster_rank() ^ 1u, at = smem_u32(act) + operand_off(act_col0 >> 3, 0, Mp), step_bytes = operand_off(2, 0, Mp);
                mbar_arrive_expect_tx(&misc->act_ready, (uint32_t)theirs * step_bytes);
                bulk_s2cluster(map_shared_rank(at, peer), at, (uint32_t)steps * step_bytes, map_shared_rank(smem_u32(&misc->act_ready), peer));
            } else if (lane == 0) {
                mbar_arrive(&misc->act_ready);
            }
            __syncwarp();
        } else {
            __syncwarp();
            if (lane == 0) mbar_arrive(&misc->act_ready);
        }
    }
}

// q|k|v: the K slices' sums meet in shared memory (`ex`, free during this phase), then norm factor, bias and rotary embedding
// finish the projection: queries go to P.q, keys and values straight into the cache at the rows' slots.  Every sum is
// complete inside its block, so nothing is reduced in L2: a barrier behind plain stores is passed 1100 cycles sooner than one
// behind reductions (2450 against 3550), and the attention step starts from finished bf16 rows.
// An item is (8 rows, token): row r < 8 of a tile and row r + 8 are the two halves of a rotary pair.
template <int HD, int MODE>
__device__ __forceinline__ void epilogue_qkv(const FwdParams& P, int layer, const Part& pt, float* ex, Misc* misc, PipePos& pos, bool& dead,
                                             int warp, int lane) {
    constexpr int HD2 = HD / 2;
    const int M = P.M, tid = warp * 32 + lane, group = warp >> 2, quarter = warp & 3;
    const int slices = pt.slices, Mp = M | 1;   // odd row stride of the exchange area: no bank conflicts
    const float inv_d = 1.f / (float)P.d;
#pragma unroll 1
    for (int p = 0; p < pt.npass; ++p, ++pos.q) {
        const int pcount = pass_count(pt, p), RR = pcount * 16, t0 = pt.tile0 + pass_start(pt, p);
        const uint32_t buf = pos.q % kAccBufs;
        // where an item's output goes and what it needs: fetched before the accumulator is there
        struct Item { float2 cs; float b0, b1, rs; __nv_bfloat16* dst; };
        auto fetch = [&](int it, Item& x) {
            const int r = it & 7, m = (it >> 3) % M, T = t0 + (it >> 3) / M;
            const int head = T / (HD / 16), i = (T % (HD / 16)) * 8 + r;
            x.rs = rsqrtf(misc->sumsq[pos.sums][m] * inv_d + P.eps);
            const float* b = P.bias ? P.bias + (size_t)layer * P.n_qkv + head * HD + i : nullptr;
            x.b0 = b ? __ldg(b) : 0.f;
            x.b1 = b ? __ldg(b + HD2) : 0.f;
            x.cs = make_float2(1.f, 0.f);
            if (head < P.n_q) x.dst = P.q + (size_t)m * (P.n_q * HD) + head * HD + i;
            int L = P.L, slot = m, at = MODE == 1 ? __ldcg(P.state + ST_DEPTH + m) : m;   // tree drafts: a row's position is its depth
            __nv_bfloat16 *kc = P.kcache, *vc = P.vcache;
            if (MODE == 2) {
                int b2 = 0;
                while (b2 + 1 < P.nseq && m >= P.seq[b2 + 1].r0) ++b2;
                L = P.seq[b2].L;
                slot = at = m - P.seq[b2].r0;
                kc = P.seq[b2].kcache;
                vc = P.seq[b2].vcache;
            }
            if (head >= P.n_q) {
                const int kvh = (head - P.n_q) % P.n_kv;
                x.dst = (head - P.n_q < P.n_kv ? kc : vc) + (((size_t)layer * P.n_kv + kvh) * P.max_seq + L + slot) * HD + i;
            }
            if (head < P.n_q + P.n_kv) x.cs = __ldg(P.rope + (size_t)(L + at) * HD2 + i);
        };
        const int items = pcount * 8 * M;
        Item first;
        if (tid < items) fetch(tid, first);
        if (!dead && !mbar_wait_bounded(&misc->tmem_full[buf], (pos.q / kAccBufs) & 1u, &misc->abort_flag, P.wait_limit_ns)) dead = true;
        dead = __any_sync(0xffffffffu, dead);
        if (!dead) {
            tc_fence_after();
            if (misc->prof_ptr && tid == 0 && p == pt.npass - 1) misc->prof_ptr[10] = global_timer_ns();
            // lanes of the accumulator: slice s * RR + row; of the columns a lane wants those of its own slice.  Where a warp's lanes
            // span two slices, the two warps that share the lanes take one each; else they take a chunk of 16 tokens each
            const uint32_t taddr = misc->tmem_base + ((uint32_t)(quarter * 32) << 16) + (slices > 1 ? kTmemStack : buf * kTmemBuf);
            const int row = quarter * 32 + lane;
            const int sl0 = (quarter * 32) / RR, sl1 = (quarter * 32 + 31) / RR;
            const bool span = sl0 != sl1;
            const int sl = span && group ? sl1 : sl0;
            const bool mine = row < slices * RR && row >= sl * RR && row < (sl + 1) * RR;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                if (h * 16 < M && (span || group == h)) {
                    float v[16];
                    tmem_ld16(taddr + (uint32_t)((sl < slices ? sl : 0) * M + h * 16), v);
#pragma unroll
                    for (int n = 0; n < 16; ++n)
                        if (mine && h * 16 + n < M) ex[row * Mp + h * 16 + n] = v[n];
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&misc->tmem_empty[buf]);  // this warp's part of the accumulators may be overwritten
        }
        named_bar_sync(2, kEpilogueWarps * 32);
        if (!dead) {
#pragma unroll 1
            for (int it = tid; it < items; it += kEpilogueWarps * 32) {
                if (it != tid) fetch(it, first);
                const int r = it & 7, m = (it >> 3) % M, tl = (it >> 3) / M;
                const float* e = ex + (tl * 16 + r) * Mp + m;
                float a = 0.f, b = 0.f;
                if (slices == 8) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) { a += e[q * RR * Mp]; b += e[(q * RR + 8) * Mp]; }
                } else {
#pragma unroll 1
                    for (int q = 0; q < slices; ++q, e += RR * Mp) { a += e[0]; b += e[8 * Mp]; }
                }
                a = a * first.rs + first.b0;
                b = b * first.rs + first.b1;
                first.dst[0] = __float2bfloat16(a * first.cs.x - b * first.cs.y);
                first.dst[HD2] = __float2bfloat16(b * first.cs.x + a * first.cs.y);
            }
        }
        if (p + 1 < pt.npass) named_bar_sync(2, kEpilogueWarps * 32);   // the exchange area is used again
    }
}

// Largest of the warp's 32 values, handed to every lane.
__device__ __forceinline__ float warp_max(float v) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
// Best logit per token row over the block: lanes, then the eight epilogue warps (through `ex`, 2 KB of shared memory).
__device__ __forceinline__ void argmax_finish(const FwdParams& P, uint8_t* ex, int warp, int lane, const Best& best, bool dead) {
    float* best_v = reinterpret_cast<float*>(ex);   // [warp][row]
    int* best_i = reinterpret_cast<int*>(best_v + kEpilogueWarps * kMaxRows);
    // two reductions per row (the value, then the lowest id that has it): written out as shuffles this was 70 KB of code that ran
    // once, 7 us behind the last pass, mostly fetching itself
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h * 16 < P.M) {
#pragma unroll
            for (int n = 0; n < 16; ++n) {
                const float v = warp_max(best.v[h][n]);
                const int i = __reduce_min_sync(0xffffffffu, best.v[h][n] == v ? best.i[h][n] : 0x7fffffff);
                if (lane == n) {
                    best_v[warp * kMaxRows + h * 16 + n] = v;
                    best_i[warp * kMaxRows + h * 16 + n] = i;
                }
            }
        }
    }
    named_bar_sync(2, kEpilogueWarps * 32);
    const int t = warp * 32 + lane;
    if (t < P.M && !dead) {
        float v = best_v[t];
        int i = best_i[t];
#pragma unroll 1
        for (int w = 1; w < kEpilogueWarps; ++w) {
            const float ov = best_v[w * kMaxRows + t];
            const int oi = best_i[w * kMaxRows + t];
            if (ov > v || (ov == v && oi < i)) { v = ov; i = oi; }
        }
        P.cand_val[(size_t)blockIdx.x * kMaxRows + t] = v;
        P.cand_idx[(size_t)blockIdx.x * kMaxRows + t] = i;
    }
}

template <int HD, int MODE, int KIND>
__device__ __forceinline__ void epilogue_phase(const FwdParams& P, int layer, uint8_t* act, uint8_t* ex, Misc* misc, PipePos& pos, bool& dead,
                                               int warp, int lane) {
    Best best;
    if (KIND == PH_QKV) {
        const Part& pt = misc->part[OP_QKV];
        if (pt.ntiles > 0 && pt.nk > 0) epilogue_qkv<HD, MODE>(P, layer, pt, reinterpret_cast<float*>(ex), misc, pos, dead, warp, lane);
    } else if (KIND == PH_LM) {
#pragma unroll
        for (int n = 0; n < kMaxRows; ++n) { best.v[n >> 4][n & 15] = -CUDART_INF_F; best.i[n >> 4][n & 15] = 0x7fffffff; }
        const Part& pt = misc->part[OP_LM];
        if (pt.ntiles > 0 && pt.nk > 0) epilogue_op<OP_LM>(P, pt, act, misc, pos, dead, warp, lane, best);
        argmax_finish(P, ex, warp, lane, best, dead);
    } else if (KIND == PH_GUD) {
        const Part &gu = misc->part[OP_GU], &dn = misc->part[OP_DOWN];
        if (gu.ntiles > 0 && gu.nk > 0) epilogue_op<OP_GU>(P, gu, act, misc, pos, dead, warp, lane, best);
        if (dn.ntiles > 0 && dn.nk > 0) epilogue_op<OP_DOWN>(P, dn, act, misc, pos, dead, warp, lane, best);
    } else {
        constexpr int op = KIND == PH_O ? OP_O : OP_RAW;
        const Part& pt = misc->part[op];
        if (pt.ntiles > 0 && pt.nk > 0) epilogue_op<op>(P, pt, act, misc, pos, dead, warp, lane, best);
    }
}

// ------------------------------------------------------------------------------------------
// Split-KV attention.  The keys [0, L + M) (the new rows' keys and values are in the cache already) are cut into S ranges of
// kps keys (a multiple of 128, at most kMaxSplits ranges); the query heads of a KV head are cut into QG groups of up to
// gh heads, a group's rows (heads x M) filling at most 64 rows (the host picks gh).
// Unit (kv head, head group, s) attends the group's rows to range s under the causal mask (row j sees new keys 0..j; in a tree
// the rows on its path) and leaves an un-normalised partial result with its running maximum and sum; the output
// projection merges them while it builds its operand.
//
// The few query rows are the N side of tcgen05.mma, the keys its 128 rows: S^T = K Q^T (lane = key, column = query row), and
// O^T = V^T P (lane = output column, column = query row).  A thread of warps 0..7 owns one key and half of the query rows:
// maxima over the 128 keys by redux and one exchange between warps, probabilities to shared memory as bf16 (the B operand of
// the second product), sums by a halving exchange of 16 shuffles.  Warp 9 issues.  Tensor memory is free in this phase: S^T
// takes columns 0..63, O^T columns 64..127.
// mma.sync tiles, which this replaces, issue m16n8k16 every 16 cycles per scheduler on this part, 1 us per 64 keys.
//
// Keys and values of a chunk of 128 keys are copied asynchronously by warps 0..7.  Rows of committed keys do not depend on
// the step: those of the first chunk are requested before the grid barrier in front of this phase, so that the phase only waits
// for its queries and the new rows.  With more chunks per range, K of the next one loads during the softmax and V behind P V.
constexpr int kLoadThreads = kEpilogueWarps * 32;   // warps 0..7 copy keys and values
constexpr int kIssueWarp = kWorkerWarps - 1;        // issues the attention's tensor-core instructions
constexpr uint32_t kTmemO = 64;                     // first column of O^T

// `keys`: of the longest sequence, new rows included.
__device__ __forceinline__ void attn_split_compute(const FwdParams& P, int keys, int& S, int& kps) {
    const int QG = (P.g + P.att_gh - 1) / P.att_gh;
    int cap = P.G / (P.n_kv * QG);
    if (cap > kMaxSplits) cap = kMaxSplits;
    if (cap < 1) cap = 1;
    kps = ((keys + cap - 1) / cap + kKeyChunk - 1) / kKeyChunk * kKeyChunk;
    S = (keys + kps - 1) / kps;
}

// What a unit works on.
struct AttnUnit {
    int M, L, r0;             // rows of its sequence, committed length, first row in the launch's buffers
    int head0, nheads;        // first query head, query heads
    int s, t_begin, nkeys;    // key range: index, first key, keys
    const __nv_bfloat16 *k, *v;   // cache of its sequence, at (layer 0, KV head, first key)
};
// MODE 0: the new rows are a chain; 1: a tree (visibility from the state block); 2: the chain of
// sequence `b` of a batched step (its rows, length and KV cache from P.seq[b]).
template <int HD, int MODE>
__device__ __forceinline__ AttnUnit attn_unit(const FwdParams& P, int b, int hk, int qg, int s) {
    AttnUnit u;
    const __nv_bfloat16 *kc = P.kcache, *vc = P.vcache;
    u.M = P.M; u.L = P.L; u.r0 = 0;
    if (MODE == 2) { u.M = P.seq[b].M; u.L = P.seq[b].L; u.r0 = P.seq[b].r0; kc = P.seq[b].kcache; vc = P.seq[b].vcache; }
    u.nheads = min(P.att_gh, P.g - qg * P.att_gh);   // the last group may hold fewer heads
    u.head0 = hk * P.g + qg * P.att_gh;
    u.s = s;
    u.t_begin = s * P.att_kps;
    u.nkeys = max(0, min(u.L + u.M, u.t_begin + P.att_kps) - u.t_begin);
    const size_t off = ((size_t)hk * P.max_seq + u.t_begin) * HD;
    u.k = kc + off;
    u.v = vc + off;
    return u;
}
// Shared memory of the attention step: query rows | values | keys, rows of 64 columns (128 bytes, 128-byte swizzle) in slabs.
template <int HD>
struct AttnShape {
    static constexpr int UNITS = HD / 8;                 // 16-byte units per row
    static constexpr int QSLAB = 64 * 128, KSLAB = kKeyChunk * 128;
    static constexpr int QBYTES = HD / 64 * QSLAB, KBYTES = HD / 64 * KSLAB;
    static_assert(QBYTES + 2 * KBYTES == kAttnBytesPerDim * HD, "attention tiles");
};
// Rows [from, to) of a chunk of keys (or values) by warps 0..7, 16-byte asynchronous copies; rows past the range are zero-filled.
template <int HD>
__device__ __forceinline__ void attn_load(const FwdParams& P, const AttnUnit& u, const __nv_bfloat16* src, int layer, int chunk, int from,
                                          int to, uint8_t* dst, int wtid) {
    using A = AttnShape<HD>;
    const __nv_bfloat16* base = src + ((size_t)layer * P.n_kv * P.max_seq + chunk * kKeyChunk) * HD;
    const int q16 = wtid % A::UNITS, left = u.nkeys - chunk * kKeyChunk;
    uint8_t* d = dst + (q16 >> 3) * A::KSLAB;
#pragma unroll
    for (int i = 0; i < kKeyChunk * A::UNITS / kLoadThreads; ++i) {
        const int key = wtid / A::UNITS + i * (kLoadThreads / A::UNITS);
        const bool valid = key < left;
        if (key >= from && key < to) cp_async_16_zfill(d + swz_unit(key, q16 & 7), base + (size_t)(valid ? key : 0) * HD + q16 * 8, valid);
    }
}
// Rows of the first chunk that may be requested before the new rows' keys are there.
__device__ __forceinline__ int attn_early_rows(const AttnUnit& u) {
    const int old = u.L - u.t_begin;   // committed keys from the range's first on
    return old >= u.nkeys ? kKeyChunk : max(0, min(old, kKeyChunk));
}

// Sums over the warp of 16 columns: lane n receives column n & 15.
__device__ __forceinline__ float warp_sum16(float (&v)[16], int lane) {
#pragma unroll
    for (int off = 8; off; off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < off; ++i) {
            const float keep = up ? v[i + off] : v[i], send = up ? v[i] : v[i + off];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 16);
}

// One unit by all worker warps.  `loaded`: rows of its first chunk requested earlier; `uses`: completions of misc->att_bar so far.
template <int HD, int MODE>
__device__ __forceinline__ void attention_unit(const FwdParams& P, Misc* misc, int layer, const AttnUnit& u, int loaded, uint8_t* att,
                                               uint8_t* Ps, int wtid, uint32_t& uses, unsigned long long* prof) {
    using A = AttnShape<HD>;
    constexpr bool TREE = MODE == 1;
    const int warp = wtid >> 5, lane = wtid & 31;
    const int M = u.M, R = u.nheads * M, RP = (R + 15) & ~15;   // R <= 64
    const uint32_t minv = 65536u / (uint32_t)M + 1u;            // row / M = row * minv >> 16 for rows below 64
    uint8_t *Qs = att, *Vs = att + A::QBYTES, *Ks = Vs + A::KBYTES;
    const int nkeys = u.nkeys, nch = (nkeys + kKeyChunk - 1) / kKeyChunk;
    if (prof && wtid == 0) prof[2] = global_timer_ns();
    // query rows (past R: zeros) and what is missing of the first chunk
    for (int un = wtid; un < RP * A::UNITS; un += kWorkerThreads) {
        const int r = un / A::UNITS, q16 = un % A::UNITS;
        const int hl = (int)((uint32_t)r * minv >> 16), j = r - hl * M;
        const bool valid = r < R;
        const __nv_bfloat16* src = P.q + (size_t)(u.r0 + (valid ? j : 0)) * (P.n_q * HD) + (u.head0 + (valid ? hl : 0)) * HD + q16 * 8;
        cp_async_16_zfill(Qs + (q16 >> 3) * A::QSLAB + swz_unit(r, q16 & 7), src, valid);
    }
    if (nch > 0 && warp < kEpilogueWarps && loaded < kKeyChunk) attn_load<HD>(P, u, u.k, layer, 0, loaded, kKeyChunk, Ks, wtid);
    cp_async_commit();
    if (nch > 0 && warp < kEpilogueWarps && loaded < kKeyChunk) attn_load<HD>(P, u, u.v, layer, 0, loaded, kKeyChunk, Vs, wtid);
    cp_async_commit();

    // this warp's keys (accumulator lanes) and query rows: columns c0 .. c0 + 16 ng - 1; lane n looks after column c0 + n
    const int quarter = warp & 3, half = warp >> 2;
    const int c0 = half ? (RP >= 48 ? 32 : 16) : 0, ng = warp >= kEpilogueWarps ? 0 : half ? max(0, (RP - c0) >> 4) : min(2, (RP >= 48 ? 32 : 16) >> 4);
    const int my_r = c0 + lane, my_h = (int)((uint32_t)my_r * minv >> 16), my_j = my_r - my_h * M;
    const uint32_t tm = misc->tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0;
    float* red = misc->att_red[warp & 7];
    float m = -CUDART_INF_F, l = 0.f;
    const int new0 = u.L - u.t_begin;   // range index of the first new key
    bool dead = *(volatile int*)&misc->abort_flag != 0;

    cp_async_wait<1>();
    fence_proxy_async_smem();
    named_bar_sync(1, kWorkerThreads);   // queries and keys are in place
    if (prof && wtid == 0) prof[3] = global_timer_ns();
#pragma unroll 1
    for (int c = 0; c < nch; ++c) {
        const int left = nkeys - c * kKeyChunk;
        if (warp == kIssueWarp) {
            tc_fence_after();
            if (elect_one()) {
                const uint32_t ka = smem_u32(Ks), qa = smem_u32(Qs), id = umma_idesc_bf16(128u, (uint32_t)RP);
#pragma unroll
                for (int ks = 0; ks < HD / 16; ++ks)
                    umma_bf16(misc->tmem_base, umma_desc_sw128(ka + (uint32_t)((ks >> 2) * A::KSLAB + (ks & 3) * 32)),
                              umma_desc_sw128(qa + (uint32_t)((ks >> 2) * A::QSLAB + (ks & 3) * 32)), id, (uint32_t)ks);
                umma_commit(&misc->att_bar);
            }
            __syncwarp();
        }
        if (warp < kEpilogueWarps) {
            // the scores are complete: K is free, and with the products before them V, P and O of the chunk before
            if (!dead && !mbar_wait_bounded(&misc->att_bar, uses & 1u, &misc->abort_flag, P.wait_limit_ns)) dead = true;
            dead = __any_sync(0xffffffffu, dead);
            tc_fence_after();
            if (prof && wtid == 0 && c == 0) prof[4] = global_timer_ns();
            if (c > 0) attn_load<HD>(P, u, u.v, layer, c, 0, kKeyChunk, Vs, wtid);
            cp_async_commit();
            if (c + 1 < nch) attn_load<HD>(P, u, u.k, layer, c + 1, 0, kKeyChunk, Ks, wtid);
            cp_async_commit();
            // columns (bit n: c0 + n) that see this thread's key
            const int kk = quarter * 32 + lane, e = c * kKeyChunk + kk - new0;
            unsigned see = kk < left ? 0xffffffffu : 0u;
            if (c * kKeyChunk + quarter * 32 + 31 >= new0) {   // a new key among the warp's
                const unsigned anc = TREE ? (unsigned)__ldcg(P.state + ST_ANC + min(my_j, kMaxRows - 1)) : 0u;
#pragma unroll 1
                for (int i = 0; i < M; ++i) {
                    const unsigned b = __ballot_sync(0xffffffffu, TREE ? ((anc >> i) & 1u) != 0 : i <= my_j);
                    if (e == i) see &= b;
                }
            }
            // maximum of every column over the 128 keys
            const float scale = P.scale_log2e;
            float mx = -CUDART_INF_F;
            if (!dead) {
#pragma unroll 1
                for (int g = 0; g < ng; ++g) {
                    float v[16];
                    tmem_ld16(tm + (uint32_t)(g * 16), v);
                    const unsigned sg = see >> (g * 16);
#pragma unroll
                    for (int n = 0; n < 16; ++n) {
                        const float x = warp_max((sg >> n) & 1u ? v[n] * scale : -CUDART_INF_F);
                        if (lane == g * 16 + n) mx = x;
                    }
                }
            }
            red[lane] = mx;
            named_bar_sync(2, kLoadThreads);
            mx = m;
#pragma unroll
            for (int w = 0; w < 4; ++w) mx = fmaxf(mx, misc->att_red[half * 4 + w][lane]);
            const float ref = mx == -CUDART_INF_F ? 0.f : mx;   // no key so far
            const float corr = exp2f(m - ref);
            m = mx;
            if (c > 0 && !dead && __any_sync(0xffffffffu, corr != 1.f)) {
                // the output so far refers to the old maximum
#pragma unroll 1
                for (int g = 0; g < ng; ++g) {
                    float v[16];
                    uint32_t o[16];
                    tmem_ld16(tm + kTmemO + (uint32_t)(g * 16), v);
#pragma unroll
                    for (int n = 0; n < 16; ++n) o[n] = __float_as_uint(v[n] * __shfl_sync(0xffffffffu, corr, g * 16 + n));
                    tmem_st16(tm + kTmemO + (uint32_t)(g * 16), o);
                }
                tmem_st_wait();
            }
            float sum = 0.f;
            if (!dead) {
                uint8_t* pd = Ps + (kk >> 6) * (RP * 128) + c0 * 128 + (kk & 7) * 2;   // row c0, column kk & 63 of its slab, without the swizzle
                const uint32_t ku = (uint32_t)((kk >> 3) & 7) << 4;
#pragma unroll 1
                for (int g = 0; g < ng; ++g) {
                    float v[16];
                    tmem_ld16(tm + (uint32_t)(g * 16), v);
                    const unsigned sg = see >> (g * 16);
#pragma unroll
                    for (int n = 0; n < 16; ++n) {
                        const float x = ex2_ftz(v[n] * scale - __shfl_sync(0xffffffffu, ref, g * 16 + n));
                        v[n] = (sg >> n) & 1u ? x : 0.f;
                        *reinterpret_cast<__nv_bfloat16*>(pd + (g * 16 + n) * 128 + (ku ^ (uint32_t)((n & 7) << 4))) = __float2bfloat16(v[n]);
                    }
                    const float t = warp_sum16(v, lane);
                    if ((lane >> 4) == g) sum = t;
                }
            }
            l = l * corr + sum;
            ++uses;
        }
        cp_async_wait<1>();   // V of this chunk
        fence_proxy_async_smem();
        tc_fence_before();
        named_bar_sync(1, kWorkerThreads);   // values and probabilities are in place
        if (warp == kIssueWarp) {
            tc_fence_after();
            if (elect_one()) {
                // heads of 64: rows 64..127 of the instruction are the keys, the tile behind V, into lanes nobody reads
                const uint32_t va = smem_u32(Vs), pa = smem_u32(Ps), id = umma_idesc_bf16(128u, (uint32_t)RP) | (1u << 15);   // A: features contiguous
                const int steps = (min(left, kKeyChunk) + 15) >> 4;
#pragma unroll 1
                for (int ks = 0; ks < steps; ++ks)
                    umma_bf16(misc->tmem_base + kTmemO, umma_desc_sw128_mn(va + (uint32_t)ks * 2048u, (uint32_t)A::KSLAB),
                              umma_desc_sw128(pa + (uint32_t)((ks >> 2) * (RP * 128) + (ks & 3) * 32)), id, (uint32_t)(c | ks));
                if (c + 1 == nch) umma_commit(&misc->att_bar);
            }
            __syncwarp();
        }
        if (c + 1 < nch) {
            cp_async_wait<0>();   // K of the next chunk
            fence_proxy_async_smem();
            named_bar_sync(1, kWorkerThreads);
        }
    }
    if (prof && wtid == 0) prof[5] = global_timer_ns();
    // un-normalised partial result of this key range
    if (warp < kEpilogueWarps) {
        red[lane] = l;
        named_bar_sync(2, kLoadThreads);
        const int row = ((u.head0 + my_h) * kMaxSplits + u.s) * kMaxRows + u.r0 + my_j;   // partial result of this lane's column
        if (quarter == 0 && lane < ng * 16 && my_r < R) {
            float sum = 0.f;
#pragma unroll
            for (int w = 0; w < 4; ++w) sum += misc->att_red[half * 4 + w][lane];
            __stcg(reinterpret_cast<float2*>(P.part_ml) + row, make_float2(m, sum));
        }
        if (nch > 0) {
            if (!dead && !mbar_wait_bounded(&misc->att_bar, uses & 1u, &misc->abort_flag, P.wait_limit_ns)) dead = true;
            dead = __any_sync(0xffffffffu, dead);
            tc_fence_after();
            ++uses;
            if (!dead && quarter * 32 < HD) {
                float* po = P.part_o + quarter * 32 + lane;
#pragma unroll 1
                for (int g = 0; g < ng; ++g) {
                    float v[16];
                    tmem_ld16(tm + kTmemO + (uint32_t)(g * 16), v);
#pragma unroll
                    for (int n = 0; n < 16; ++n) {
                        const int rw = __shfl_sync(0xffffffffu, row, g * 16 + n);
                        if (c0 + g * 16 + n < R) __stcg(po + (size_t)rw * HD, v[n]);
                    }
                }
            }
            tc_fence_before();
        }
    }
}

// `early`: rows of the first chunk of the block's first unit that were requested before the grid barrier.
template <int HD, int MODE>
__device__ __forceinline__ void attention_phase(const FwdParams& P, Misc* misc, int layer, int early, uint8_t* smem, int wtid, uint32_t& uses,
                                                unsigned long long* prof) {
    const int per_seq = P.att_per_seq, QG = P.att_QG, S = P.att_S;
    const int nunits = per_seq * (MODE == 2 ? P.nseq : 1);
#pragma unroll 1
    for (int unit = blockIdx.x; unit < nunits; unit += P.G) {
        int b = P.att_b0, hk = P.att_hk0, qg = P.att_qg0, s = P.att_s0;
        if (unit != (int)blockIdx.x) {  // further units of this block (more units than blocks: batched steps)
            const int u = unit % per_seq, rem = u % (QG * S);
            b = unit / per_seq;
            hk = u / (QG * S);
            qg = rem / S;
            s = rem % S;
            early = 0;
        }
        // batched: every sequence takes the key ranges of the longest one; a range past its own length holds no key
        attention_unit<HD, MODE>(P, misc, layer, attn_unit<HD, MODE>(P, b, hk, qg, s), early, smem + P.u_off, smem + P.p_off, wtid, uses, prof);
        named_bar_sync(1, kWorkerThreads);  // the unit's shared-memory tiles are free again
        if (prof && wtid == 0) { prof[6] = global_timer_ns(); prof[7] = (unsigned long long)(s + 1 == S); }
    }
}
// Before the grid barrier in front of the attention phase: requests the committed keys of the first chunk of the block's unit.  Only
// once the block's own products of the phase before have completed (their operand lies where the keys go), which
// warps 0..7 know from their epilogue.
template <int HD, int MODE>
__device__ __forceinline__ int attention_early(const FwdParams& P, int layer, uint8_t* att, int wtid) {
    using A = AttnShape<HD>;
    if ((int)blockIdx.x >= P.att_per_seq * (MODE == 2 ? P.nseq : 1)) return 0;
    const AttnUnit u = attn_unit<HD, MODE>(P, P.att_b0, P.att_hk0, P.att_qg0, P.att_s0);
    if (u.nkeys <= 0) return 0;
    const int n = attn_early_rows(u);
    if ((wtid >> 5) < kEpilogueWarps) {
        attn_load<HD>(P, u, u.v, layer, 0, 0, n, att + A::QBYTES, wtid);
        attn_load<HD>(P, u, u.k, layer, 0, 0, n, att + A::QBYTES + A::KBYTES, wtid);
    }
    cp_async_commit();
    return n;
}
// ------------------------------------------------------------------------------------------
__device__ void embed_phase(const FwdParams& P, const DraftArg& draft, int wtid) {
    if (blockIdx.x == 0 && draft.n >= 0) {
        // the caller's draft becomes the one of the state block, for the kernels behind this one
        if (wtid < draft.n) P.state[ST_DRAFT + wtid] = draft.tok[wtid];
        if (wtid == 0) {
            P.state[ST_DRAFT_LEN] = draft.n;
            P.state[ST_BASE_LEN] = draft.n;
            P.state[ST_SEG_USED] = 0;
            P.state[ST_TREE_ON] = 0;
        }
    }
    // residual rows from the embedding table; rows beyond M are cleared
    const int units = kMaxRows * (P.d / 8);
#pragma unroll 1
    for (int u = blockIdx.x * kWorkerThreads + wtid; u < units; u += P.G * kWorkerThreads) {
        const int row = u / (P.d / 8), c8 = u % (P.d / 8);
        float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
        if (row < P.M) {
            int tok;
            if (P.mode == 1) tok = P.hist[P.L + row];
            else if (row == 0) tok = P.state[ST_PENDING];
            else if (draft.n >= 0) tok = draft.tok[row - 1];
            else tok = (row <= P.state[ST_DRAFT_LEN]) ? P.state[ST_DRAFT + row - 1] : 0;
            tok = min(max(tok, 0), P.V - 1);
            const uint4 raw = __ldg(reinterpret_cast<const uint4*>(P.emb + (size_t)tok * P.d + c8 * 8));
            const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&raw);
            const float2 f0 = __bfloat1622float2(pb[0]), f1 = __bfloat1622float2(pb[1]);
            const float2 f2 = __bfloat1622float2(pb[2]), f3 = __bfloat1622float2(pb[3]);
            lo = make_float4(f0.x, f0.y, f1.x, f1.y);
            hi = make_float4(f2.x, f2.y, f3.x, f3.y);
        }
        float* dst = P.h + (size_t)row * P.d + c8 * 8;
        __stcg(reinterpret_cast<float4*>(dst), lo);
        __stcg(reinterpret_cast<float4*>(dst + 4), hi);
    }
}
// ------------------------------------------------------------------------------------------
// One GEMM phase as seen by the worker warps: build the token operand, then the tensor-core
// thread walks the block's stages while the epilogue warps drain the accumulators.
template <int HD, int MODE, int KIND>
__device__ __forceinline__ void gemm_phase(const FwdParams& P, int layer, NormPrep& prep, uint8_t* smem, Misc* misc, PipePos& pos, int wtid,
                                           unsigned long long* prof) {
    constexpr int op = KIND == PH_QKV ? OP_QKV : KIND == PH_O ? OP_O : KIND == PH_GUD ? OP_GU : KIND == PH_LM ? OP_LM : OP_RAW;
    const int warp = wtid >> 5, lane = wtid & 31;
    uint8_t* U = smem + P.u_off;
    const Part& p0 = misc->part[op];
    const bool have0 = p0.ntiles > 0 && p0.nk > 0;
    bool dead = *(volatile int*)&misc->abort_flag != 0;
    if (wtid == 0) misc->prof_ptr = prof;
    if (have0) {
        if (!dead) {
            if (KIND == PH_O) {
                if (P.att_S <= 20 && P.M * p0.nk * 2 > kWorkerThreads / 4) build_merged_operand<2, 10>(P, p0, U, wtid);
                else if (P.att_S <= 20) build_merged_operand<4, 5>(P, p0, U, wtid);
                else build_merged_operand<4, kMaxSplits / 4>(P, p0, U, wtid);
            } else {
                build_norm_operand<KIND>(P, prep, layer, U, misc, pos.sums, wtid);
            }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&misc->op_ready);   // this warp's part of the operand may be read by the tensor core
    }
    if (prof && wtid == 0) prof[2] = global_timer_ns();
    if (warp < kEpilogueWarps) {
        // the rows' sums of squares the epilogue scales with come from all builder warps
        if (have0 && !dead && !mbar_wait_bounded(&misc->op_ready, pos.ops & 1u, &misc->abort_flag, P.wait_limit_ns)) dead = true;
        PipePos ep = pos;
        epilogue_phase<HD, MODE, KIND>(P, layer, smem + P.act_off, smem + P.p_off, misc, ep, dead, warp, lane);
        if (prof && wtid == 0) prof[4] = global_timer_ns();
    }
    // pipeline positions advance identically for every role (a worker only follows accumulator passes and operands)
    if (have0) {
        ++pos.ops;
        if (KIND != PH_O) pos.sums ^= 1u;
        pos.q += (uint32_t)p0.npass;
    }
    if (KIND == PH_GUD) {
        const Part& dn = misc->part[OP_DOWN];
        if (dn.ntiles > 0 && dn.nk > 0) pos.q += (uint32_t)dn.npass;
    }
}

// The tensor-core thread: all operations of the launch in order.  It waits for operands, never for grid barriers.
__device__ __forceinline__ void mma_loop(const FwdParams& P, uint8_t* smem, Misc* misc) {
    PipePos pos;
    pos.slot = pos.par = pos.q = pos.ops = pos.sums = pos.w_full = pos.w_acc = 0;
    uint32_t act_uses = 0;
    bool ready = false;
    const uint32_t ring0 = smem_u32(smem);
    const uint64_t wait_limit = P.wait_limit_ns;
    int ph = P.ph_begin;
    auto run = [&](int op) {   // one operation once its token operand is complete
        const Part& pt = misc->part[op];
        if (pt.ntiles == 0 || pt.nk == 0) return true;
        const bool down = op == OP_DOWN;
        unsigned long long* prof = P.prof ? P.prof + ((size_t)(ph - P.ph_begin) * P.G + blockIdx.x) * kProfWords : nullptr;
        if (!down) pos.w_full = pos.w_acc = 0;
        const long long t0 = clock64();
        const bool ok = mma_op(P, op, ring0, misc, pos, ready, down ? &misc->act_ready : &misc->op_ready, (down ? act_uses++ : pos.ops++) & 1u);
        if (prof) {
            prof[9] = (unsigned long long)(clock64() - t0);  // cycles from turning to the operation (the phase's last one) to its last instruction
            prof[op == OP_GU ? 5 : 3] = global_timer_ns();
            prof[7] = pos.w_full;
            prof[8] = pos.w_acc;
        }
        return ok;
    };
    // q|k|v, o, gate|up, down of every layer (phases 0, 2, 3 and 3 of the layer), then the LM head; or one operation alone
    const int lm = 1 + kPhasesPerLayer * P.n_layers, nops = ph == 0 ? 4 * P.n_layers + (P.ph_end > lm ? 1 : 0) : (P.ph_end > lm ? 1 : 0);
    const int first = ph == 0 ? 0 : ph == lm ? OP_LM : OP_RAW;
#pragma unroll 1
    for (int i = 0; i < nops; ++i) {
        int op = first;
        if (first == 0) {
            op = i < 4 * P.n_layers ? i & 3 : (int)OP_LM;
            ph = op == OP_LM ? lm : 1 + kPhasesPerLayer * (i >> 2) + (op == 0 ? 0 : op < 3 ? op + 1 : 3);
        }
        if (!run(op)) break;
    }
    // all tensor-core work must have completed before tensor memory is returned
    umma_commit(&misc->done_bar);
    mbar_wait_bounded(&misc->done_bar, 0, &misc->abort_flag, wait_limit);
}

// ------------------------------------------------------------------------------------------
// Where a wait was abandoned in one of a pair's blocks, nobody may have waited for the other one's last columns.  One thread of each block gets here,
// behind a cluster barrier (all that will be sent has been), and keeps its block there: the two tell each other in how many phases they have
// sent, wait for what they have been sent, and leave once the other one has done so.  Every wait has the usual limit.
__device__ __noinline__ void leave_pair(const FwdParams& P, Misc* misc) {
    const uint32_t other = cluster_rank() ^ 1u;
    auto tell = [&](int* word, uint32_t v) { st_release_cluster_u32(map_shared_rank(smem_u32(word), other), v); };
    auto hear = [&](int* word) {
        const uint64_t t0 = global_timer_ns();
        uint32_t v;
        while ((v = ld_acquire_cluster_u32(smem_u32(word))) == 0u && global_timer_ns() - t0 < P.wait_limit_ns) {}
        return v;
    };
    // gate|up is a layer's last phase and a phase is skipped only where all behind it are: whole layers
    int mine = P.ph_begin == 0 && misc->part[OP_DOWN].nk > 0 ? P.n_layers : 0;
    if (mine > 0 && *(volatile int*)&misc->abort_flag) {
        int per_layer = 0;
        for (int op = OP_QKV; op <= OP_DOWN; ++op) per_layer += misc->part[op].npass;
        mine = min(mine, *(volatile int*)&misc->pair_passes / per_layer);
    }
    tell(&misc->pair_theirs, (uint32_t)mine + 1u);
    const uint32_t theirs = hear(&misc->pair_theirs);
    const int debt = theirs ? pair_debt(mine, (int)theirs - 1) : PAIR_NONE;
    const bool last = !(debt & PAIR_LAST) || mbar_drain(&misc->act_ready, (uint32_t)(mine - 1) & 1u, P.wait_limit_ns);
    if (last && (debt & PAIR_NEXT)) {
        mbar_arrive_expect_tx(&misc->act_ready, (uint32_t)(misc->part[OP_DOWN].nk - misc->part[OP_GU].ntiles / 2) * operand_off(2, 0, operand_rows(P, P.M, 1)));
        for (int w = 1; w < kEpilogueWarps; ++w) mbar_arrive(&misc->act_ready);
        mbar_drain(&misc->act_ready, (uint32_t)mine & 1u, P.wait_limit_ns);
    }
    tell(&misc->pair_done, 1u);
    hear(&misc->pair_done);
}

// ------------------------------------------------------------------------------------------
// HD: head dimension; MODE: chain, tree or batch (see attention_unit), or 3: the stand-alone GEMM alone (a launch of its own).
template <int HD, int MODE>
__global__ void __launch_bounds__(kThreads, 1) sdv_forward_kernel(const __grid_constant__ FwdParams Pg, const __grid_constant__ DraftArg draft) {
    static_assert(sizeof(FwdParams) % 4 == 0, "parameter block is copied word by word");
    extern __shared__ __align__(1024) uint8_t smem[];   // the launch's only shared memory: starts on a 1024-byte boundary
    Misc* misc = reinterpret_cast<Misc*>(smem + kMiscOff);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (Pg.l_from_state && Pg.state[ST_BUDGET] == 0) {
        // a step enqueued behind the end of its run: nothing to do, but the barrier counter moves as the host assumed
        if (tid == 0 && Pg.ph_end - Pg.ph_begin > 1) red_release_add_u32(Pg.bar, (unsigned)(Pg.ph_end - Pg.ph_begin - 1));
        return;
    }
    {
        const int* src = reinterpret_cast<const int*>(&Pg);
        int* dst = reinterpret_cast<int*>(&misc->P);
        for (int i = tid; i < (int)(sizeof(FwdParams) / 4); i += kThreads) dst[i] = src[i];
    }
    __syncthreads();
    const FwdParams& P = misc->P;
    if (tid == 0) {
        // Rows past the draft the device holds would be padding: they are not computed.  The shared-memory plan follows the
        // rows (fewer rows leave room for more ring slots).
        FwdParams& Q = misc->P;
        if (Pg.rows_from_state) {
            Q.M = min(Pg.M, Pg.state[ST_DRAFT_LEN] + 1);
            Q.att_gh = Pg.att_gh_rows[Q.M - 1];
        }
        Q.NB = Q.M > 16 ? 32 : 16;
        plan_smem_rows(Q, Q.M);
    }
    if (tid >= 32 && tid < 32 + OP_COUNT) misc->part[tid - 32] = get_part(Pg.op[tid - 32], Pg.op[OP_GU], blockIdx.x, Pg.G);

    if (tid == 0) {
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(&misc->full[s], 1);
            mbar_init(&misc->empty[s], 1);
        }
        for (int b = 0; b < (int)kAccBufs; ++b) {
            mbar_init(&misc->tmem_full[b], 1);
            mbar_init(&misc->tmem_empty[b], kEpilogueWarps);
        }
        mbar_init(&misc->op_ready, kBuilderWarps);
        mbar_init(&misc->act_ready, kEpilogueWarps);
        mbar_init(&misc->att_bar, 1);
        mbar_init(&misc->done_bar, 1);
        misc->abort_flag = 0;
        misc->skip = 0;
        misc->pair_abort = misc->pair_theirs = misc->pair_done = 0;
        for (int r = 0; r < kMaxRows; ++r) misc->sumsq[0][r] = 0.f;
        mbar_fence_init();
    }
    if (warp == kMmaWarp) tmem_alloc(&misc->tmem_base, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (MODE != 3) cluster_arrive();   // this block's barriers are there
    if (tid == 0) {
        if (Pg.l_from_state) misc->P.L = Pg.state[ST_KV_LEN];
        // the block's first attention unit: the same for every layer, so its index arithmetic is done here
        FwdParams& Q = misc->P;
        int keys = Q.L + Q.M;
        if (MODE == 2) {
            keys = 1;
            for (int b = 0; b < Q.nseq; ++b) keys = max(keys, Q.seq[b].L + Q.seq[b].M);
        }
        attn_split_compute(Q, keys, Q.att_S, Q.att_kps);
        const int S = Q.att_S;
        Q.att_QG = (Q.g + Q.att_gh - 1) / Q.att_gh;
        Q.att_per_seq = Q.n_kv * Q.att_QG * S;
        const int unit = blockIdx.x, u = unit % Q.att_per_seq, rem = u % (Q.att_QG * S);
        Q.att_b0 = unit / Q.att_per_seq;
        Q.att_hk0 = u / (Q.att_QG * S);
        Q.att_qg0 = rem / S;
        Q.att_s0 = rem % S;
    }

    if (tid >= 32 && tid < 32 + OP_COUNT) {
        const int op = tid - 32;
        misc->shape[op] = norm_shape(P, misc->part[op]);
        misc->mma[op] = mma_shape(P, misc->part[op], smem_u32(smem + (op == OP_DOWN ? P.act_off : P.u_off)));
    }
    __syncthreads();
    if (MODE != 3) cluster_wait();
    // A block leaves once the other one of its pair no longer copies from or to it: each has waited for the other's columns before it gets here
    // unless a wait was abandoned, and then one thread stays until they are there.
    auto finish = [&]() {
        if (MODE != 3) {
            __syncwarp();
            cluster_sync();
        }
    };

    if (warp == kProducerWarp) {
        if (lane == 0) producer_loop(P, smem, misc);
        finish();
        return;
    }
    if (warp == kMmaWarp) {
        if (elect_one()) mma_loop(P, smem, misc);
        __syncwarp();
        tc_fence_before();
        named_bar_sync(3, kWorkerThreads + 32);   // the workers have read the last accumulators
        tc_fence_after();
        tmem_dealloc(misc->tmem_base, kTmemCols);
        finish();
        if (MODE != 3 && lane == 0 && P.op[OP_DOWN].P_row == 2 && (*(volatile int*)&misc->abort_flag | *(volatile int*)&misc->pair_abort) != 0) leave_pair(P, misc);
        return;
    }

    const int wtid = tid;  // 0 .. kWorkerThreads-1
    PipePos pos;
    pos.slot = pos.par = pos.q = pos.ops = pos.sums = pos.w_full = pos.w_acc = 0;
    uint32_t att_uses = 0;
    int ph = P.ph_begin;
    unsigned target = P.bar_base;
    bool skip = false;   // after an abandoned wait the remaining phases do no work but still meet at every barrier
    unsigned long long* pp = nullptr;
    auto enter = [&]() {
        pp = P.prof ? P.prof + ((size_t)(ph - P.ph_begin) * P.G + blockIdx.x) * kProfWords : nullptr;
        if (pp && wtid == 0) pp[0] = global_timer_ns();
    };
    auto leave = [&]() {
        ++ph;
        if (pp) {
            named_bar_sync(1, kWorkerThreads);
            if (wtid == 0) pp[1] = global_timer_ns();
        }
    };
    // the grid barrier behind a phase; `prepare` works out what the next one needs
    auto meet = [&](auto prepare) {
        target += (unsigned)P.G;
        skip = grid_barrier(P, target, misc, wtid, prepare);
    };
    const int n_layers = P.n_layers, lm = 1 + kPhasesPerLayer * n_layers;
    NormPrep prep;
    if (MODE == 3) {
        norm_prep<PH_RAW>(prep, P, misc, 0, wtid, 0);
        enter();
        gemm_phase<HD, MODE, PH_RAW>(P, 0, prep, smem, misc, pos, wtid, pp);
        leave();
    } else {
        if (ph == 0) {
            enter();
            embed_phase(P, draft, wtid);
            leave();
#pragma unroll 1
            for (int layer = 0; layer < n_layers; ++layer) {
                int early = 0;
                meet([&]() { norm_prep<PH_QKV>(prep, P, misc, layer, wtid, 0); });
                enter();
                if (!skip) gemm_phase<HD, MODE, PH_QKV>(P, layer, prep, smem, misc, pos, wtid, pp);
                leave();
                meet([&]() { early = attention_early<HD, MODE>(P, layer, smem + P.u_off, wtid); });
                enter();
                if (!skip) attention_phase<HD, MODE>(P, misc, layer, early, smem, wtid, att_uses, pp);
                leave();
                meet([]() {});
                enter();
                if (!skip) gemm_phase<HD, MODE, PH_O>(P, layer, prep, smem, misc, pos, wtid, pp);
                leave();
                meet([&]() { norm_prep<PH_GUD>(prep, P, misc, layer, wtid, 0); });
                enter();
                if (!skip) gemm_phase<HD, MODE, PH_GUD>(P, layer, prep, smem, misc, pos, wtid, pp);
                leave();
            }
            if (ph < P.ph_end) meet([&]() { norm_prep<PH_LM>(prep, P, misc, 0, wtid, 0); });
        } else if (ph == lm) {
            norm_prep<PH_LM>(prep, P, misc, 0, wtid, 0);
        }
        if (ph == lm && ph < P.ph_end) {
            enter();
            if (!skip) gemm_phase<HD, MODE, PH_LM>(P, 0, prep, smem, misc, pos, wtid, pp);
            leave();
        }
    }
    tc_fence_before();
    named_bar_sync(3, kWorkerThreads + 32);
    if (*(volatile int*)&misc->abort_flag) {   // final by now: the tensor-core thread is done, so the streamer is or was told
        if (wtid == 0) {
            atomicExch(P.state + ST_ERR, 1);
            if (MODE != 3 && P.op[OP_DOWN].P_row == 2) {
                misc->pair_passes = (int)pos.q;
                st_release_cluster_u32(map_shared_rank(smem_u32(&misc->pair_abort), cluster_rank() ^ 1u), 1u);
            }
        }
    }
    finish();
}

}  // namespace sdv
