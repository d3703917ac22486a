// C-ABI of the verify-path library (see include/sdv.h): context set-up, the static work
// partition, weight re-layout, and the launch sequences of prefill / draft / verify / commit.
#include "../../include/sdv.h"

#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <new>
#include <vector>

#include "dense.cuh"
#include "device_once.h"
#include "forward.cuh"
#include "layout.cuh"
#include "small_gemm.cuh"
#include "small_kernels.cuh"

using namespace sdv;

namespace {

constexpr int kPinnedBytes = 4096;   // a context's page-locked memory
inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

struct Regions {
    size_t state, bstate, bar, never, hist, db, rope, norm_w, bias, wlayers, wlm, emb, kcache, vcache, h, q, part_o,
        part_ml, cand_val, cand_idx, logits, raw_out, staging, wraw, xstage, prof, succ, occ, dw, dlm, dh, dxn, dpart, dq, datt, dact, total;
    size_t layer_stride, staging_bytes, raw_kmax;
};

bool config_ok(const sdv_config* c) {
    if (!c) return false;
    if (c->n_layers < 1 || c->d_model < 64 || c->d_model % 64 || c->d_ffn < 64 || c->d_ffn % 64) return false;
    if (c->vocab < 16 || c->vocab % 16) return false;
    if (c->head_dim != 64 && c->head_dim != 128) return false;
    if (c->n_kv_heads < 1 || c->n_q_heads < 1 || c->n_q_heads % c->n_kv_heads) return false;
    const int g = c->n_q_heads / c->n_kv_heads;
    if (g > 8) return false;
    if (c->k_max < 1 || c->k_max > SDV_K_MAX) return false;
    if (c->max_seq < c->k_max + 2) return false;
    if (c->ngram_n < 1 || c->ngram_n > SDV_NGRAM_MAX || c->ngram_min < 1 || c->ngram_min > c->ngram_n) return false;
    if (!(c->rope_theta > 0.f) || !(c->rms_eps > 0.f)) return false;
    return true;
}

// `own_weights` false: a context that reads another context's weights carves none of the weight regions
// (nor the staging areas only weight loading and the stand-alone GEMM use).
Regions carve(const sdv_config* c, bool own_weights = true) {
    Regions r;
    memset(&r, 0, sizeof(r));
    const size_t d = c->d_model, f = c->d_ffn, V = c->vocab, hd = c->head_dim;
    const size_t nq = (size_t)c->n_q_heads * hd, nkv = (size_t)c->n_kv_heads * hd, nqkv = nq + 2 * nkv;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off = align_up(off + bytes, 256);
        return o;
    };
    auto take_w = [&](size_t bytes) { return take(own_weights ? bytes : 0); };
    r.state = take(ST_WORDS * 4);
    r.bstate = take(ST_WORDS * 4);  // state block a batched verify step runs on
    r.bar = take(256);
    r.never = take(256);
    r.hist = take(((size_t)c->max_seq + 64) * 4);
    r.db = take(((size_t)c->max_seq + 64) * 4);
    r.rope = take_w((size_t)c->max_seq * (hd / 2) * sizeof(float2));
    r.norm_w = take_w(((size_t)c->n_layers * 2 + 1) * d * 4);
    r.bias = take_w((size_t)c->n_layers * nqkv * 4);
    r.layer_stride = (nqkv * d + d * nq + 2 * f * d + d * f) * 2;
    r.wlayers = take_w(r.layer_stride * c->n_layers);
    r.wlm = take_w(V * d * 2);
    r.emb = take_w(V * d * 2);
    const size_t kvb = (size_t)c->n_layers * c->n_kv_heads * c->max_seq * hd * 2;
    r.kcache = take(kvb);
    r.vcache = take(kvb);
    r.h = take((size_t)kMaxRows * d * 4);
    r.q = take((size_t)kMaxRows * nq * 2);
    size_t raw_kmax = f;  // the stand-alone GEMM takes operands of any K up to max(f, d, nq)
    if (d > raw_kmax) raw_kmax = d;
    if (nq > raw_kmax) raw_kmax = nq;
    r.raw_kmax = raw_kmax;
    r.part_o = take((size_t)c->n_q_heads * kMaxSplits * kMaxRows * hd * 4);
    r.part_ml = take((size_t)c->n_q_heads * kMaxSplits * kMaxRows * 2 * 4);
    r.cand_val = take((size_t)kMaxGrid * kMaxRows * 4);
    r.cand_idx = take((size_t)kMaxGrid * kMaxRows * 4);
    r.logits = take((size_t)kMaxRows * V * 4);
    size_t st = 2 * f * d * 2;  // gate | up of one layer, the largest per-layer group
    if (nqkv * d * 2 > st) st = nqkv * d * 2;
    if (d * nq * 2 > st) st = d * nq * 2;
    if (st < ((size_t)64 << 20)) st = (size_t)64 << 20;
    r.staging_bytes = st;
    r.staging = take_w(st);
    r.wraw = take_w(st);
    r.raw_out = take_w((size_t)kMaxRows * (st / 128) * 4);  // N <= staging / (2 bytes * 64 columns)
    r.xstage = take((size_t)kMaxRows * raw_kmax * 4);
    r.prof = take((size_t)(3 + kPhasesPerLayer * c->n_layers) * kMaxGrid * kProfWords * 8);
    // dense prefill path: row-major weight copies (a tied LM head is the embedding itself) and the activations of one
    // sub-chunk; the partial sums of a product's K shares and the calibration's per-tile best logits share a region
    r.dw = take_w(r.layer_stride * c->n_layers);
    r.dlm = c->tied_lm_head ? r.emb : take_w(V * d * 2);
    r.dh = take((size_t)kDenseMaxRows * d * 4);
    r.dxn = take((size_t)kDenseMaxRows * d * 2);
    size_t dp = (size_t)(kMaxGrid / 2) * 256 * 256 * 4;                                    // K shares: one tile per pair of SMs at most (the best logits are fewer)
    const size_t one = (size_t)kDenseMaxRows * (nqkv > d ? nqkv : d) * 4;                  // a product without K shares
    if (one > dp) dp = one;
    r.dpart = take(dp);
    r.dq = take((size_t)kDenseMaxRows * nq * 2);
    r.datt = take((size_t)kDenseMaxRows * nq * 2);
    r.dact = take((size_t)kDenseMaxRows * f * 2);
    r.succ = take((size_t)c->max_seq * SDV_CALIB_MAX * 4);  // calibration: sampled successors per context position
    r.occ = take((size_t)c->max_seq * SDV_CALIB_MAX * 4);   // and where each occurs in the context
    r.total = off;
    return r;
}

// Chooses how an operation's grid of row tiles x column steps is cut among the blocks and how a
// block walks its share (RW row tiles per pass, SK column steps per stage).  Model of a block's
// time in microseconds: streaming its share at a fair share of HBM bandwidth or walking its
// stages and passes, whichever is longer, plus building its token operand (the bytes it reads from
// L2: residual rows, or split-KV partial results when `merge`) and, when partial sums meet in L2
// (column partitions, or the residual add), the reductions of all blocks.
void choose_partition(OpDesc& o, int G, int rows, bool merge, bool always_add) {
    double best_t = -1.0;
    o.RW = 16;
    o.SK = kStageBytes / kStepBytes / 16;
    o.P_row = 1;
    o.P_k = 1;
    o.unit = 1;
    o.follow = 0;
    for (int RW = 16; RW >= 1; RW /= 2) {
        const int SK = kStageBytes / kStepBytes / RW;
        for (int pr = 1; pr <= o.T && pr <= G; ++pr) {
            const int pk_max = G / pr < o.K16 ? G / pr : o.K16;
            for (int pk = 1; pk <= pk_max; ++pk) {
                const int tiles = (o.T + pr - 1) / pr, ks = (o.K16 + pk - 1) / pk;
                const int passes = (tiles + RW - 1) / RW;
                const int stages = passes * ((ks + SK - 1) / SK);
                const double stream = (double)tiles * ks * kStepBytes / 44000.0;
                const double walk = 0.06 * stages + 0.25 * passes;
                const double operand_bytes =
                    merge ? (double)rows * ks * 2 * 21 * 40.0 : (double)rows * ks * 16 * 4.0;
                double t = (stream > walk ? stream : walk) + 0.8 + operand_bytes / 60000.0;
                if (pk > 1 || always_add) t += 0.7 + 0.016 * pk * (rows / 9.0);
                if (best_t < 0 || t < best_t - 1e-9) {
                    best_t = t;
                    o.RW = RW;
                    o.SK = SK;
                    o.P_row = pr;
                    o.P_k = pk;
                }
            }
        }
    }
}
// A block whose share has fewer row tiles than a pass may hold walks it in one pass all the same:
// RW then only sets the stage length.  Shrinking RW to the tiles a block really has (a power of two)
// doubles SK until a stage is back at the ring slot's size, i.e. fewer, longer bulk copies.
void fit_pass_width(OpDesc& o) {
    if (o.follow) return;
    const int per = o.unit * ((o.T / o.unit + o.P_row - 1) / o.P_row);  // row tiles of the largest share
    while (o.RW > 1 && o.RW / 2 >= per) o.RW /= 2;
    o.SK = kStageBytes / kStepBytes / o.RW;
}

// Operations whose epilogue needs complete sums: all columns in one block, rows spread evenly.
void full_k_partition(OpDesc& o, int G, int unit) {
    o.RW = 16;
    o.SK = kStageBytes / kStepBytes / 16;
    o.unit = unit;
    o.follow = 0;
    o.P_k = 1;
    o.P_row = o.T / unit < G ? o.T / unit : G;
}

// q|k|v: all columns in one block as well (its epilogue finishes the projection).  A share is a tile or a few, so eighths (or
// quarters, halves) of its columns are stacked to fill the instruction's 128 rows.
void stacked_partition(OpDesc& o, int G) {
    full_k_partition(o, G, 1);
    const int per = (o.T + o.P_row - 1) / o.P_row;   // row tiles of the largest share
    o.slices = 8;
    while (o.slices > 1 && (o.slices * per > 8 || o.K16 % o.slices)) o.slices /= 2;
    o.RW = 8 / o.slices;                             // one accumulator per pass
    while (o.RW > 1 && o.RW / 2 >= per) o.RW /= 2;
    o.SK = kStageBytes / kStepBytes / (o.RW * o.slices);
}

// Shared-memory plan of a launch over `rows` token rows (plan_smem_rows), and whether they fit.
struct SmemPlan {
    int NG, NB, nstage, u_bytes;
    bool ok;
};
SmemPlan plan_smem(FwdParams& P, int rows, bool raw_only) {
    P.plan_ks = P.plan_act = P.plan_attn = 0;
    for (int i = 0; i < OP_COUNT; ++i) {
        const OpDesc& o = P.op[i];
        if (o.T == 0 || o.follow || (raw_only != (i == OP_RAW))) continue;
        const int ks = (o.K16 + o.P_k - 1) / o.P_k;
        if (ks > P.plan_ks) P.plan_ks = ks;
    }
    if (!raw_only) {
        const OpDesc& gu = P.op[OP_GU];
        P.plan_act = P.op[OP_DOWN].P_row * ((gu.T / gu.unit + gu.P_row - 1) / gu.P_row);
        P.plan_attn = kAttnBytesPerDim * P.hd;
    }
    plan_smem_rows(P, rows);
    SmemPlan s;
    s.NG = (rows + 7) / 8;
    s.NB = rows > 16 ? 32 : 16;
    s.nstage = P.nstage;
    s.u_bytes = P.act_off - P.u_off;
    s.ok = P.nstage >= 2 && P.plan_act * 32 * rows <= kActSmemMax;
    return s;
}

// What pairs must not cost, whose down projection's operand is twice as large, for any number of rows (a batched step has more than k_max + 1) and of
// heads per attention unit, of which a launch chooses one: a launch that fits with single blocks, or the third ring slot.  Two slots hold the stream up:
// layers of the 7B shape, pairs on two slots against single blocks on three, 16 rows 13 % slower at 256 and 2048 keys and 11 % at 8192, 17 rows 13 and
// 10 %; at the numbers of rows where they have as many slots the two are within 0.6 %.  A fourth slot is worth less than the pairs mostly give: 3B
// shape, 15 rows, pairs on three against four 0.7 to 1.1 % faster (14 and 16 rows, as many slots: 2.8 to 4 %); 0.5B, 32 rows, four against five 5.3 to 5.5 %.
bool pairs_fit(const FwdParams& P, int g) {
    FwdParams one = P, two = P;
    one.op[OP_DOWN].P_row = 1;
    two.op[OP_DOWN].P_row = 2;
    for (int rows = 1; rows <= kMaxRows; ++rows)
        for (int gh = 1; gh <= g; ++gh) {
            one.att_gh = two.att_gh = gh;
            const SmemPlan a = plan_smem(one, rows, false), b = plan_smem(two, rows, false);
            if ((a.ok && !b.ok) || (a.nstage >= 3 && b.nstage < 3)) return false;
        }
    return true;
}

// The operations of one layer, in streaming order, and the LM head: shapes, partitions, offsets.  may_pair: blocks may come in pairs.
void setup_ops(FwdParams& P, const sdv_config* cfg, int G, bool may_pair) {
    const int d = cfg->d_model, f = cfg->d_ffn, hd = cfg->head_dim;
    const int nq = cfg->n_q_heads * hd, nkv = cfg->n_kv_heads * hd, nqkv = nq + 2 * nkv;
    struct { int idx, N, K; } ops[5] = {{OP_QKV, nqkv, d}, {OP_O, d, nq}, {OP_GU, 2 * f, d}, {OP_DOWN, d, f},
                                        {OP_LM, cfg->vocab, d}};
    unsigned long long woff = 0;
    int rot = 0;
    const int rows_max = cfg->k_max + 1;
    for (int i = 0; i < 5; ++i) {
        OpDesc& o = P.op[ops[i].idx];
        memset(&o, 0, sizeof(o));
        o.T = ops[i].N / 16;
        o.K16 = ops[i].K / 16;
        switch (ops[i].idx) {
            case OP_QKV: stacked_partition(o, G); break;
            case OP_O: choose_partition(o, G, rows_max, true, true); break;
            case OP_GU: full_k_partition(o, G, 2); break;   // pairs of tiles: 16 SwiGLU columns = one column step of down
            case OP_LM: full_k_partition(o, G, 1); break;
            default: {  // down: every block multiplies the SwiGLU columns it produced, or a pair of blocks those of both
                const OpDesc& gu = P.op[OP_GU];
                o.RW = 16; o.SK = kStageBytes / kStepBytes / 16; o.unit = 1; o.follow = 1;
                // In pairs each block has half of the rows, so half as many partial sums meet in L2, which the phase waits for: gate|up + down 12.6
                // -> 12.0 us at 9 rows of the 1.5B shape, 19.1 -> 16.5 at 32, 29.1 -> 25.0 at 17 rows of the 3B shape, 7.4 -> 6.5 at 9 of the 0.5B
                // shape.  A launch in clusters takes 2 us more, so the sums have to be many: with two layers 16 K (256 columns x 64 shares) lose 1.6 us of
                // a launch of 53.5, with 24 layers 133 K (896 x 148) gain 21 of 593.  With 16 layers (5 to 32 rows, 512 keys) all that was tried gains:
                // above the line, 64 K to 133 K sums, 0.7 to 9.3 %; below it, 32 K to 61 K, 1.3 to 5.9 % and 16 K 0.4 to 1.7 %, so the line is on the
                // safe side for models of few layers.  The blocks of a pair are those of a cluster: an even number of shares, beginning at an
                // even block; the operand of both shares takes half of kActSmemMax at most, and must not cost a number of rows that single blocks
                // can take, nor the third ring slot (pairs_fit).
                const int steps = (gu.T / gu.unit + gu.P_row - 1) / gu.P_row;
                const bool pairs = may_pair && G % 2 == 0 && gu.P_row % 2 == 0 && gu.rot % 2 == 0 && o.T >= 2 && 16 * o.T * gu.P_row >= kPairSums &&
                                   2 * steps * 32 * (rows_max | 1) <= kActSmemMax / 2;
                o.P_row = pairs ? 2 : 1;
                o.P_k = gu.P_row / o.P_row;
                break;
            }
        }
        if (ops[i].idx == OP_GU && G % 2 == 0) rot += rot % 2;
        if (ops[i].idx != OP_QKV) fit_pass_width(o);
        if (ops[i].idx == OP_DOWN) {
            o.rot = P.op[OP_GU].rot;
        } else {
            o.rot = rot % G;
            rot += o.P_row * o.P_k;
        }
        o.w_off = (ops[i].idx == OP_LM) ? 0 : woff;
        if (ops[i].idx != OP_LM) woff += (unsigned long long)ops[i].N * ops[i].K * 2;
    }
    OpDesc& down = P.op[OP_DOWN];
    if (down.P_row == 2 && !pairs_fit(P, cfg->n_q_heads / cfg->n_kv_heads)) {
        down.P_row = 1;
        down.P_k = P.op[OP_GU].P_row;
    }
}

// The grid, one persistent block per SM, and its operations.  Pairs of blocks are clusters of one launch, which needs all of them at once: where
// the device cannot hold them (`clusters_held`: how many it can), or the shape does not take pairs, the blocks are single ones on every SM.
template <typename F>
int setup_grid(FwdParams& P, const sdv_config* cfg, int sms, F clusters_held) {
    const int even = sms & ~1;
    if (even >= 2) {
        setup_ops(P, cfg, even, true);
        if (P.op[OP_DOWN].P_row == 2 ? clusters_held() >= even / 2 : even == sms) return even;
    }
    setup_ops(P, cfg, sms, false);
    return sms;
}

}  // namespace

struct sdv_ctx {
    sdv_config cfg;
    uint8_t* ws;
    size_t ws_bytes;
    Regions r;
    cudaStream_t stream;
    int G;
    FwdParams P;  // template; per-launch fields are filled at launch
    int* pinned;  // page-locked copy of the state block, then room for the tokens of a run
    cudaEvent_t ev0, ev1;
    // host mirror of the device state
    int kv_len, hist_len, n_ctx;
    bool prefill_done, weights_loaded, verified, draft_pending;
    int draft_k;    // k of the pending sdv_draft
    int last_rows;  // rows of the last verify at most (a draft on the device may have been shorter)
    unsigned bar_base;  // grid-barrier counter value before the next launch (wraps; only differences are used)
    int parity;
    int profile;
    int last_cuda;
    long long launches;
    bool have_verify_time;
    bool poisoned;
    std::vector<CUtensorMap>* maps;  // dense path, see MapIndex
    bool dense_ok;       // the tensor maps could be built (else every chunk takes the small-row path)
    int calib_b;         // successors sampled per context position during prefill (0: calibration off)
    bool calibrated;     // the calibration tables cover the whole context
    bool tree_pending;   // the device draft is a tree
    bool tree_verified;  // the outstanding verify result is a tree's
    std::vector<cudaEvent_t>* run_ev;  // event pairs around the forward kernels of the last run of enqueued steps
    int run_steps;       // steps of that run
    sdv_ctx* leader;     // the context whose weights this one reads (nullptr: its own)
    const float* logits_src;  // where the rows of this context's last verify step lie (a batched step leaves them in the first context's buffer)
};

namespace {

int cuda_fail(sdv_ctx* ctx, cudaError_t e) {
    if (ctx) ctx->last_cuda = (int)e;
    return SDV_ECUDA;
}
#define CK(call)                                          \
    do {                                                  \
        cudaError_t e_ = (call);                          \
        if (e_ != cudaSuccess) return cuda_fail(ctx, e_); \
    } while (0)

typedef void (*ForwardKernel)(const FwdParams, const DraftArg);
// The kind of launch the forward kernel is compiled for: chain, tree, batch, or the stand-alone GEMM alone (whatever the heads).
int forward_mode(const FwdParams& P) { return P.ph_begin == 2 + kPhasesPerLayer * P.n_layers ? 3 : P.nseq > 0 ? 2 : P.tree ? 1 : 0; }
// The forward kernel compiled for this launch's head dimension and kind.
ForwardKernel forward_kernel(const FwdParams& P) {
    static const ForwardKernel table[2][4] = {{sdv_forward_kernel<64, 0>, sdv_forward_kernel<64, 1>, sdv_forward_kernel<64, 2>, sdv_forward_kernel<64, 3>},
                                              {sdv_forward_kernel<128, 0>, sdv_forward_kernel<128, 1>, sdv_forward_kernel<128, 2>, sdv_forward_kernel<64, 3>}};
    return table[P.hd == 128][forward_mode(P)];
}
// The kernel may use all shared memory (an attribute of each device).
cudaError_t size_kernel(const FwdParams& P) {
    static DeviceOnce sized[2][4];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = sized[P.hd == 128][forward_mode(P)].run(
            dev, [&]() { return cudaFuncSetAttribute(forward_kernel(P), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget); });
    return e;
}
// A launch in pairs of blocks, together on the device where `together`.
struct PairLaunch {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[2];
    PairLaunch(const PairLaunch&) = delete;
    PairLaunch(int G, cudaStream_t stream, bool together) {
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3(G);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kSmemBudget;
        cfg.stream = stream;
        memset(at, 0, sizeof(at));
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        at[1].id = cudaLaunchAttributeCooperative;
        at[1].val.cooperative = 1;
        cfg.attrs = at;
        cfg.numAttrs = together ? 2 : 1;
    }
};
// Pairs of blocks of the forward kernel that the device holds at once (all its kinds have the same launch shape).
int pairs_held(const FwdParams& P) {
    const PairLaunch l(P.G, nullptr, false);
    int n = 0;
    if (size_kernel(P) == cudaSuccess && cudaOccupancyMaxActiveClusters(&n, (const void*)forward_kernel(P), &l.cfg) == cudaSuccess) return n;
    cudaGetLastError();   // not to be reported by the next check: single blocks need no answer
    return 0;
}
cudaError_t launch_kernel(const FwdParams& P, const DraftArg* draft, cudaStream_t stream) {
    const ForwardKernel k = forward_kernel(P);
    const cudaError_t e = size_kernel(P);
    if (e != cudaSuccess) return e;
    DraftArg none;
    none.n = -1;
    void* args[] = {(void*)&P, (void*)(draft ? draft : &none)};
    if (forward_mode(P) == 3) return cudaLaunchKernel((const void*)k, dim3(P.G), dim3(kThreads), args, kSmemBudget, stream);
    // Phases meet at grid barriers, so more than one phase needs all blocks co-resident.
    if (P.op[OP_DOWN].P_row != 2) {
        if (P.ph_end - P.ph_begin > 1)
            return cudaLaunchCooperativeKernel((const void*)k, dim3(P.G), dim3(kThreads), args, kSmemBudget, stream);
        return cudaLaunchKernel((const void*)k, dim3(P.G), dim3(kThreads), args, kSmemBudget, stream);
    }
    // pairs of blocks share the down projection
    const PairLaunch l(P.G, stream, P.ph_end - P.ph_begin > 1);
    return cudaLaunchKernelExC(&l.cfg, (const void*)k, args);
}

bool apply_plan(FwdParams& P, int rows, bool raw_only) {
    if (!raw_only && P.att_gh < 1) P.att_gh = rows >= 64 ? 1 : 64 / rows;   // not chosen yet: room for any choice
    const SmemPlan sp = plan_smem(P, rows, raw_only);
    P.M = rows;
    P.NB = sp.NB;
    return sp.ok;
}

// Attention split of a launch: heads per unit (a unit's rows, heads x M, fill at most 64); the key ranges follow (as in
// attn_split_compute).  Cost of a choice in units of about 0.15 us: per round of one unit per block a fixed price, and per
// chunk of 128 keys the latency of its products and exchanges and the softmax of its query rows, 16 at a time.
int plan_attention(const FwdParams& P, int rows, int L, int nseq) {
    int best = -1, best_gh = 1;
    for (int gh = 1; gh <= P.g; ++gh) {
        if (gh * rows > 64 && gh > 1) break;
        const int QG = (P.g + gh - 1) / gh, RP = (gh * rows + 15) / 16;
        int cap = P.G / (P.n_kv * QG);
        if (cap > kMaxSplits) cap = kMaxSplits;
        if (cap < 1) cap = 1;
        const int keys = L + rows, chunks = ((keys + cap - 1) / cap + kKeyChunk - 1) / kKeyChunk, S = (keys + chunks * kKeyChunk - 1) / (chunks * kKeyChunk);
        const int rounds = (P.n_kv * QG * S * nseq + P.G - 1) / P.G;
        const int cost = rounds * (6 + chunks * (4 + RP));
        if (best < 0 || cost <= best) {  // ties: more heads per unit (fewer reloads of the keys)
            best = cost;
            best_gh = gh;
        }
    }
    return best_gh;
}

// `batch`: the sequences of a batched step (then `rows` is their total, `L` the longest length, and the launch
// reads its tokens from the batch state block).
struct BatchPlan {
    int n, max_rows;
    BatchSeq seq[kMaxBatch];
};
int launch_forward(sdv_ctx* ctx, int rows, int L, int mode, int ph_begin, int ph_end, bool timed, bool force_logits = false,
                   bool tree = false, const BatchPlan* batch = nullptr, bool l_from_state = false, cudaEvent_t* run_ev = nullptr,
                   const DraftArg* draft = nullptr) {
    FwdParams P = ctx->P;
    P.l_from_state = l_from_state ? 1 : 0;
    const bool raw_only = (ph_begin == 2 + kPhasesPerLayer * ctx->cfg.n_layers);
    // A draft on the device may be shorter than `rows` allows: its own rows alone are computed.  In parity mode every row is, the
    // padding (token 0) too, so that what is stored for the rows past the draft never dates from another step.
    P.rows_from_state = (mode == 0 && !batch && !draft && !ctx->parity) ? 1 : 0;
    P.L = L;
    P.att_gh = P.g < 1 ? 1 : plan_attention(P, batch ? batch->max_rows : rows, L, batch ? batch->n : 1);
    if (P.rows_from_state)   // for every number of rows the draft may turn out to have
        for (int r = 1; r <= rows; ++r) P.att_gh_rows[r - 1] = (uint8_t)plan_attention(P, r, L, 1);
    if (!apply_plan(P, rows, raw_only)) return SDV_EINVAL;
    P.nseq = 0;
    if (batch) {
        P.nseq = batch->n;
        for (int b = 0; b < batch->n; ++b) P.seq[b] = batch->seq[b];
        P.state = (int*)(ctx->ws + ctx->r.bstate);
    }
    ctx->logits_src = P.logits;
    P.mode = mode;
    P.ph_begin = ph_begin;
    P.ph_end = ph_end;
    P.bar_base = ctx->bar_base;
    P.store_logits = (ctx->parity || force_logits) ? 1 : 0;
    P.tree = tree ? 1 : 0;
    P.prof = ctx->profile ? (unsigned long long*)(ctx->ws + ctx->r.prof) : nullptr;
    const int nbar = ph_end - ph_begin - 1;
    ctx->bar_base += (unsigned)(nbar * ctx->G);
    if (timed) CK(cudaEventRecord(run_ev ? run_ev[0] : ctx->ev0, ctx->stream));
    cudaError_t e = launch_kernel(P, draft, ctx->stream);
    if (e != cudaSuccess) return cuda_fail(ctx, e);
    ctx->launches++;
    if (timed) {
        CK(cudaEventRecord(run_ev ? run_ev[1] : ctx->ev1, ctx->stream));
        if (!run_ev) ctx->have_verify_time = true;
    }
    return SDV_OK;
}

// `published`: the last kernel has written the state block to the page-locked copy itself.
int read_state(sdv_ctx* ctx, bool published = false) {
    if (!published) CK(cudaMemcpyAsync(ctx->pinned, ctx->ws + ctx->r.state, ST_WORDS * 4, cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    if (ctx->pinned[ST_ERR] == 1) {
        ctx->poisoned = true;
        return SDV_ETIMEOUT;
    }
    return SDV_OK;
}

// Drafts (or tree nodes) of the outstanding verify step: what the device verified, which may be fewer than the host's bound
// allowed for.  Their rows, and the pending token's, are the ones it computed.
int verified_drafts(sdv_ctx* ctx, int* n) {
    int rc = read_state(ctx);
    if (rc) return rc;
    const int dl = ctx->pinned[ST_DRAFT_LEN];
    *n = dl < ctx->last_rows - 1 ? dl : ctx->last_rows - 1;
    return SDV_OK;
}

int pack_op(sdv_ctx* ctx, const OpDesc& o, uint8_t* dst_base, const uint16_t* s0, int rows0, const uint16_t* s1,
            int rows1, const uint16_t* s2, int K, int mode, int t_begin, int t_end, int row_base) {
    const long long total = (long long)(t_end - t_begin) * 16 * (K / 8);
    int blocks = (int)((total + 255) / 256);
    if (blocks > 148 * 16) blocks = 148 * 16;
    pack_weights_kernel<<<blocks, 256, 0, ctx->stream>>>(o, ctx->P.op[OP_GU], dst_base, s0, rows0, s1, rows1, s2, K, mode,
                                                       t_begin, t_end, row_base, ctx->cfg.head_dim);
    ctx->launches++;
    CK(cudaGetLastError());
    return SDV_OK;
}

void fill_draft_arg(DraftArg& a, const int32_t* tok, int n) {
    memset(&a, 0, sizeof(a));
    a.n = n;
    for (int i = 0; i < n; ++i) a.tok[i] = tok[i];
}

int commit_common(sdv_ctx* ctx, int max_emit, int force_accept, int force_token, int32_t* host_emitted, int* n_emitted,
                  int* kv_len) {
    int* hist = (int*)(ctx->ws + ctx->r.hist);
    if (ctx->tree_verified) {
        // the accepted path's K/V rows move to consecutive cache slots before the length advances
        kv_compact_kernel<<<dim3(ctx->cfg.n_layers * ctx->cfg.n_kv_heads, 2), 128, 0, ctx->stream>>>(
            ctx->P.state, ctx->P.kcache, ctx->P.vcache, ctx->cfg.max_seq, ctx->cfg.head_dim, max_emit);
        ctx->launches++;
        ctx->tree_verified = false;
    }
    commit_kernel<<<1, 64, 0, ctx->stream>>>(ctx->P.state, hist, max_emit, force_accept, force_token, ctx->pinned);
    ctx->launches++;
    CK(cudaGetLastError());
    int rc = read_state(ctx, true);
    if (rc) return rc;
    const int n = ctx->pinned[ST_N_EMITTED];
    ctx->kv_len = ctx->pinned[ST_KV_LEN];
    ctx->hist_len = ctx->pinned[ST_HIST_LEN];
    ctx->verified = false;
    ctx->draft_pending = false;
    ctx->tree_pending = false;
    if (n_emitted) *n_emitted = n;
    if (kv_len) *kv_len = ctx->kv_len;
    if (host_emitted)
        for (int i = 0; i < n; ++i) host_emitted[i] = ctx->pinned[ST_EMITTED + i];
    return SDV_OK;
}

// ---- dense prefill path (csrc/dense.cuh)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn() {
    static std::atomic<EncodeTiledFn> fn{nullptr};   // the same for every thread and device
    EncodeTiledFn known = fn.load(std::memory_order_acquire);
    if (!known) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess) {
            known = (EncodeTiledFn)p;
            fn.store(known, std::memory_order_release);
        }
    }
    return known;
}
// bf16 matrix [rows][K] row-major on this GPU; box = box_rows x 64 columns, 128-byte swizzle, zeros outside.
bool make_map(CUtensorMap* m, const void* base, uint64_t rows, uint64_t K, uint32_t box_rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {K, rows};
    const cuuint64_t strides[1] = {K * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kDenseBK, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// Tensor maps of a context: activations (normalised rows, attention output, SwiGLU output), key and value cache, the LM head, then per layer
// q|k|v, o, gate|up and down with boxes of 64 rows (tiles of 128 features) and again with boxes of 128 (256 features).
enum MapIndex { MAP_XN = 0, MAP_ATT, MAP_ACT, MAP_K, MAP_V, MAP_LM, MAP_LAYERS };
inline size_t map_at(int layer, int matrix, int bn) { return MAP_LAYERS + 8 * (size_t)layer + 2 * matrix + (bn == 256 ? 1 : 0); }

// A launch that may overlap the tail of the kernel before it (programmatic dependent launch), in clusters of `cluster`
// blocks along x when > 0 (0: as the kernel declares).
template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(sdv_ctx* ctx, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, unsigned cluster, Args... args) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = ctx->stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 0 ? 2 : 1;
    ctx->launches++;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// How a product of M x N outputs is cut: features per tile and K shares.  Model of its time in microseconds: rounds of
// one tile per pair of SMs, each its K stages (64 columns: 0.26 us with 128 features, 0.40 with 256) and a fixed price, and
// the fp32 partial sums, written here and read by the next kernel, each way at 6 TB/s (6e6 bytes per us).
struct DensePlan {
    int bn, splits;
};
DensePlan plan_dense(const sdv_ctx* ctx, int M, int N, int K, bool may_split) {
    const int pairs = ctx->G / 2, mt = (M + 255) / 256, nkb = K / kDenseBK;
    DensePlan best = {256, 1};
    double best_t = -1.0;
    for (int bn = 128; bn <= 256; bn *= 2) {
        const int nt = (N + bn - 1) / bn;
        for (int sp = 1; sp <= (may_split ? kDenseMaxSplits : 1) && sp <= nkb; ++sp) {
            if (sp > 1 && mt * nt * sp > pairs) break;
            const int rounds = (mt * nt * sp + pairs - 1) / pairs;
            double t = rounds * (((nkb + sp - 1) / sp) * (bn == 256 ? 0.40 : 0.26) + 1.0);
            if (may_split) t += 2.0 * sp * (double)M * N * 4.0 / 6.0e6;
            if (best_t < 0 || t < best_t - 1e-9) {
                best_t = t;
                best.bn = bn;
                best.splits = sp;
            }
        }
    }
    return best;
}

template <int EPI, int BN>
cudaError_t launch_dense_tiles(sdv_ctx* ctx, const CUtensorMap& a, const CUtensorMap& b, int M, int N, int K, int splits, float* part,
                               __nv_bfloat16* out_bf16, int ld_bf16, DenseTopOut top) {
    const int tiles = ((M + 255) / 256) * ((N + BN - 1) / BN) * splits, pairs = ctx->G / 2;
    return launch_dependent(ctx, dense_gemm_kernel<EPI, BN>, dim3(2 * (tiles < pairs ? tiles : pairs)), dim3(kDenseThreads<EPI>),
                            DenseShape<BN>::kSmemBytes, 0, a, b, M, N, K, splits, part, out_bf16, ld_bf16, top, ctx->P.state + ST_ERR,
                            2000000000ull);
}
// Product of the activations behind `a` with one of a layer's matrices into partial sums; *splits receives their number.
cudaError_t dense_product(sdv_ctx* ctx, MapIndex a, int layer, int matrix, int M, int N, int K, int* splits) {
    const std::vector<CUtensorMap>& m = *ctx->maps;
    const DensePlan pl = plan_dense(ctx, M, N, K, true);
    float* part = (float*)(ctx->ws + ctx->r.dpart);
    *splits = pl.splits;
    if (pl.bn == 256)
        return launch_dense_tiles<EPI_PARTIAL, 256>(ctx, m[a], m[map_at(layer, matrix, 256)], M, N, K, pl.splits, part, nullptr, 0, DenseTopOut());
    return launch_dense_tiles<EPI_PARTIAL, 128>(ctx, m[a], m[map_at(layer, matrix, 128)], M, N, K, pl.splits, part, nullptr, 0, DenseTopOut());
}

// The dense path's kernels may use the shared memory their shapes need (an attribute of each device).
cudaError_t dense_attributes() {
    static DeviceOnce once;
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    return once.run(dev, []() {
        constexpr auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
        cudaError_t e = cudaFuncSetAttribute(dense_gemm_kernel<EPI_PARTIAL, 128>, attr, DenseShape<128>::kSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(dense_gemm_kernel<EPI_PARTIAL, 256>, attr, DenseShape<256>::kSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(dense_gemm_kernel<EPI_SWIGLU, 256>, attr, DenseShape<256>::kSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(dense_gemm_kernel<EPI_TOP, 256>, attr, DenseShape<256>::kSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(dense_attention_kernel<128>, attr, DenseAttShape<128>::kSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(dense_attention_kernel<64>, attr, DenseAttShape<64>::kSmemBytes);
        return e;
    });
}

// One sub-chunk of `rows` (1..kDenseMaxRows) context tokens at positions L..L+rows-1 through every layer:
// fills their K/V rows.  The tokens are hist[L .. L+rows).  The last row's residual is also left where the LM head of
// the forward kernel reads row 0; with `succ` the best logits of every row (calibration) go to succ[row][calib_b].
int dense_prefill_rows(sdv_ctx* ctx, int rows, int L, int* succ) {
    const sdv_config& c = ctx->cfg;
    const int d = c.d_model, f = c.d_ffn, hd = c.head_dim, nq = c.n_q_heads * hd, nkv = c.n_kv_heads * hd, nqkv = nq + 2 * nkv;
    uint8_t* ws = ctx->ws;
    float* h = (float*)(ws + ctx->r.dh);
    float* part = (float*)(ws + ctx->r.dpart);
    __nv_bfloat16* xn = (__nv_bfloat16*)(ws + ctx->r.dxn);
    __nv_bfloat16* q = (__nv_bfloat16*)(ws + ctx->r.dq);
    __nv_bfloat16* att = (__nv_bfloat16*)(ws + ctx->r.datt);
    __nv_bfloat16* act = (__nv_bfloat16*)(ws + ctx->r.dact);
    const int* hist = (const int*)(ws + ctx->r.hist);
    const std::vector<CUtensorMap>& maps = *ctx->maps;
    const float* norm_w = ctx->P.norm_w;
    const float* bias = ctx->P.bias;
    const int g = ctx->P.g;
    CK(dense_attributes());
    // rows: four columns per thread and turn
    const int turns = d <= 2048 ? 1 : d <= 4096 ? 2 : 4;
    int nt = ((turns <= 2 ? d / 4 / turns : d / 4) + 31) / 32 * 32;
    if (nt > 1024) nt = 1024;
    const auto norm_kernel = turns == 1 ? dense_residual_norm_kernel<1> : turns == 2 ? dense_residual_norm_kernel<2> : dense_residual_norm_kernel<4>;
    // four rotary pairs per thread, q|k|v of a row in one turn where a block can hold them
    int ft = (nqkv / 8 + 31) / 32 * 32;
    if (ft > 1024) ft = 1024;
    // attention: the queries whose g heads fill a 128-row tile; key shares so that the blocks fill the chip once (clusters of
    // more than two leave some SMs of a group of 18 or 20 unused, hence 7/8) and keep two blocks of 128 keys each, one per stream
    const int QR = 128 / g, qtiles = (rows + QR - 1) / QR;
    int cs = ctx->G * 7 / 8 / (qtiles * c.n_kv_heads);
    if (cs > 8) cs = 8;
    if (cs > (L + rows + 255) / 256) cs = (L + rows + 255) / 256;
    if (cs < 1) cs = 1;
    int splits = 0;
    CK(launch_dependent(ctx, norm_kernel, dim3(rows), dim3(nt), 0, 0, hist + L, ctx->P.emb, c.vocab, h, part, 0, norm_w, xn, d,
                        c.rms_eps, nullptr));
    for (int l = 0; l < c.n_layers; ++l) {
        const size_t layer_off = (size_t)l * c.n_kv_heads * c.max_seq * hd;
        const bool last = l + 1 == c.n_layers;
        CK(dense_product(ctx, MAP_XN, l, 0, rows, nqkv, d, &splits));
        CK(launch_dependent(ctx, dense_qkv_finish_kernel, dim3(rows), dim3(ft), 0, 0, part, splits, bias ? bias + (size_t)l * nqkv : nullptr,
                            ctx->P.rope, q, c.n_q_heads, c.n_kv_heads, hd, ctx->P.kcache, ctx->P.vcache, layer_off, c.max_seq, L));
        CK(launch_dependent(ctx, hd == 128 ? dense_attention_kernel<128> : dense_attention_kernel<64>, dim3(qtiles * cs, c.n_kv_heads),
                            dim3(kDenseAttThreads), hd == 128 ? DenseAttShape<128>::kSmemBytes : DenseAttShape<64>::kSmemBytes, (unsigned)cs,
                            maps[MAP_K], maps[MAP_V], q, l * c.n_kv_heads * c.max_seq, c.max_seq, c.n_q_heads, g, QR, rows, L,
                            ctx->P.scale_log2e, att, ctx->P.state + ST_ERR, 2000000000ull));
        CK(dense_product(ctx, MAP_ATT, l, 1, rows, d, nq, &splits));
        CK(launch_dependent(ctx, norm_kernel, dim3(rows), dim3(nt), 0, 0, nullptr, ctx->P.emb, c.vocab, h, part, splits,
                            norm_w + (size_t)(2 * l + 1) * d, xn, d, c.rms_eps, nullptr));
        CK((launch_dense_tiles<EPI_SWIGLU, 256>(ctx, maps[MAP_XN], maps[map_at(l, 2, 256)], rows, 2 * f, d, 1, nullptr, act, f, DenseTopOut())));
        CK(dense_product(ctx, MAP_ACT, l, 3, rows, d, f, &splits));
        // the next layer's first norm, behind the last layer the final norm (norm_w holds them in this order)
        CK(launch_dependent(ctx, norm_kernel, dim3(rows), dim3(nt), 0, 0, nullptr, ctx->P.emb, c.vocab, h, part, splits,
                            norm_w + (size_t)(2 * l + 2) * d, xn, d, c.rms_eps, last ? ctx->P.h : nullptr));
    }
    if (succ) {
        DenseTopOut top;
        const int mt = (rows + 255) / 256, tiles = mt * ((c.vocab + 255) / 256), pairs = tiles < ctx->G / 2 ? tiles : ctx->G / 2;
        const int shares = kDenseHalves<EPI_TOP> * (pairs / mt);
        top.val = part;
        top.idx = (int*)(part + (size_t)rows * shares * kDenseTopMax);
        CK((launch_dense_tiles<EPI_TOP, 256>(ctx, maps[MAP_XN], maps[MAP_LM], rows, c.vocab, d, 1, nullptr, nullptr, 0, top)));
        CK(launch_dependent(ctx, dense_top_merge_kernel, dim3(rows), dim3(256), 0, 0, top, shares, ctx->calib_b, succ));
    }
    CK(cudaGetLastError());
    return SDV_OK;
}

}  // namespace

extern "C" {

const char* sdv_strerror(int code) {
    switch (code) {
        case SDV_OK: return "ok";
        case SDV_EINVAL: return "invalid argument or unsupported shape";
        case SDV_ENOMEM: return "workspace too small";
        case SDV_ECAPACITY: return "KV cache or history capacity exceeded";
        case SDV_ESTATE: return "call not valid in the current state";
        case SDV_ECUDA: return "CUDA runtime error";
        case SDV_ETIMEOUT: return "a bounded device-side wait ran out";
        case SDV_ETOOBIG: return "problem larger than the no-allocation entry point takes";
        default: return "unknown error";
    }
}

size_t sdv_workspace_bytes(const sdv_config* cfg) {
    if (!config_ok(cfg)) return 0;
    return carve(cfg).total;
}

int sdv_last_cuda_error(const sdv_ctx* ctx) { return ctx ? ctx->last_cuda : 0; }
long long sdv_launch_count(const sdv_ctx* ctx) { return ctx ? ctx->launches : 0; }
int sdv_kv_len(const sdv_ctx* ctx) { return ctx ? ctx->kv_len : SDV_EINVAL; }

}  // extern "C"

namespace {
// A context over `dev_workspace`; with a `leader` it reads that context's weights instead of holding its own.
int create_context(const sdv_config* cfg, void* dev_workspace, size_t bytes, cudaStream_t stream, sdv_ctx* leader, sdv_ctx** out) {
    if (!out) return SDV_EINVAL;
    *out = nullptr;
    if (!config_ok(cfg) || !dev_workspace || ((uintptr_t)dev_workspace & 255)) return SDV_EINVAL;
    if (bytes < carve(cfg, leader == nullptr).total) return SDV_ENOMEM;
    sdv_ctx* ctx = new (std::nothrow) sdv_ctx();
    if (!ctx) return SDV_ENOMEM;
    memset(ctx, 0, sizeof(*ctx));
    ctx->cfg = *cfg;
    ctx->ws = (uint8_t*)dev_workspace;
    ctx->ws_bytes = bytes;
    ctx->stream = stream;
    ctx->leader = leader;
    int sms = 0, dev = 0, coop = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e != cudaSuccess || sms <= 0 || !coop) {
        delete ctx;
        return SDV_ECUDA;
    }
    if (sms > kMaxGrid) sms = kMaxGrid;
    ctx->r = carve(cfg, leader == nullptr);
    // every failure below leaves through this: what was created so far is released
    auto fail = [&](int code) {
        if (ctx->pinned) cudaFreeHost(ctx->pinned);
        if (ctx->ev0) cudaEventDestroy(ctx->ev0);
        if (ctx->ev1) cudaEventDestroy(ctx->ev1);
        delete ctx;
        return code;
    };
    e = cudaHostAlloc((void**)&ctx->pinned, kPinnedBytes, cudaHostAllocDefault);
    if (e == cudaSuccess) e = cudaEventCreate(&ctx->ev0);
    if (e == cudaSuccess) e = cudaEventCreate(&ctx->ev1);
    if (e != cudaSuccess) return fail(SDV_ECUDA);

    const int d = cfg->d_model, f = cfg->d_ffn, hd = cfg->head_dim;
    const int nq = cfg->n_q_heads * hd, nkv = cfg->n_kv_heads * hd, nqkv = nq + 2 * nkv;
    FwdParams& P = ctx->P;
    P.n_layers = cfg->n_layers; P.d = d; P.n_q = cfg->n_q_heads; P.n_kv = cfg->n_kv_heads; P.hd = hd; P.f = f;
    P.V = cfg->vocab; P.max_seq = cfg->max_seq; P.g = cfg->n_q_heads / cfg->n_kv_heads; P.n_qkv = nqkv;
    P.eps = cfg->rms_eps;
    P.scale_log2e = (float)((1.0 / sqrt((double)hd)) * 1.4426950408889634);
    if (leader) {  // its weights are laid out for its grid
        ctx->G = leader->G;
        memcpy(P.op, leader->P.op, sizeof(P.op));
    } else {
        ctx->G = setup_grid(P, cfg, sms, [&]() { P.G = sms & ~1; return pairs_held(P); });
    }
    P.G = ctx->G;
    const int rows_max = cfg->k_max + 1;
    P.layer_stride = ctx->r.layer_stride;
    uint8_t* ws = ctx->ws;
    if (leader) {
        P.wlayers = leader->P.wlayers;
        P.wlm = leader->P.wlm;
        P.wraw = nullptr;  // no stand-alone GEMM on a context without weight regions
        P.emb = leader->P.emb;
        P.norm_w = leader->P.norm_w;
        P.bias = leader->P.bias;
    } else {
        P.wlayers = ws + ctx->r.wlayers;
        P.wlm = ws + ctx->r.wlm;
        P.wraw = ws + ctx->r.wraw;
        P.emb = (const __nv_bfloat16*)(ws + ctx->r.emb);
        P.norm_w = (const float*)(ws + ctx->r.norm_w);
        P.bias = cfg->qkv_bias ? (const float*)(ws + ctx->r.bias) : nullptr;
    }
    P.rope = leader ? leader->P.rope : (const float2*)(ws + ctx->r.rope);
    P.kcache = (__nv_bfloat16*)(ws + ctx->r.kcache);
    P.vcache = (__nv_bfloat16*)(ws + ctx->r.vcache);
    P.h = (float*)(ws + ctx->r.h);
    P.q = (__nv_bfloat16*)(ws + ctx->r.q);
    P.part_o = (float*)(ws + ctx->r.part_o);
    P.part_ml = (float*)(ws + ctx->r.part_ml);
    P.cand_val = (float*)(ws + ctx->r.cand_val);
    P.cand_idx = (int*)(ws + ctx->r.cand_idx);
    P.logits = (float*)(ws + ctx->r.logits);
    P.raw_out = (float*)(ws + ctx->r.raw_out);
    P.raw_x = (const float*)(ws + ctx->r.xstage);
    P.raw_N = 0;
    P.raw_K = 0;
    P.state = (int*)(ws + ctx->r.state);
    P.hist = (const int*)(ws + ctx->r.hist);
    P.bar = (unsigned*)(ws + ctx->r.bar);
    P.wait_limit_ns = 2000000000ull;
    {
        // the widest verify step must fit the shared-memory plan
        FwdParams probe = P;
        if (!apply_plan(probe, rows_max, false)) return fail(SDV_EINVAL);
    }

    // rotary table in double, rounded once to fp32 (a follower reads its leader's)
    if (!leader) {
        const size_t n = (size_t)cfg->max_seq * (hd / 2);
        std::vector<float2> tab(n);
        for (int i = 0; i < hd / 2; ++i) {
            const double inv = pow((double)cfg->rope_theta, -2.0 * (double)i / (double)hd);
            for (int p = 0; p < cfg->max_seq; ++p) {
                const double a = (double)p * inv;
                tab[(size_t)p * (hd / 2) + i] = make_float2((float)cos(a), (float)sin(a));
            }
        }
        e = cudaMemcpyAsync(ws + ctx->r.rope, tab.data(), n * sizeof(float2), cudaMemcpyHostToDevice, ctx->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(ws + ctx->r.state, 0, ST_WORDS * 4, ctx->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws + ctx->r.bstate, 0, ST_WORDS * 4, ctx->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws + ctx->r.bar, 0, 256, ctx->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws + ctx->r.never, 0, 256, ctx->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ws + ctx->r.hist, 0, ((size_t)cfg->max_seq + 64) * 4, ctx->stream);
    // activations: h .. part_ml are contiguous regions
    if (e == cudaSuccess) e = cudaMemsetAsync(ws + ctx->r.h, 0, ctx->r.cand_val - ctx->r.h, ctx->stream);
    if (e == cudaSuccess) {
        fill_f32_kernel<<<8, 256, 0, ctx->stream>>>(P.cand_val, -INFINITY, (long long)kMaxGrid * kMaxRows);
        fill_i32_kernel<<<8, 256, 0, ctx->stream>>>(P.cand_idx, 0x7fffffff, (long long)kMaxGrid * kMaxRows);
        ctx->launches += 2;
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) return fail(SDV_ECUDA);
    // dense prefill path: tensor maps over its activation buffers and its weight copies
    ctx->maps = new (std::nothrow) std::vector<CUtensorMap>(MAP_LAYERS + 8 * (size_t)cfg->n_layers);
    ctx->dense_ok = ctx->maps != nullptr && ctx->G >= 2 && d <= 16384;  // its products run on pairs of SMs; four turns of 1024 threads x 4 columns in the row-wise kernels
    if (ctx->dense_ok && leader) {  // the weight copies of the dense path are the leader's as well
        ctx->dense_ok = leader->dense_ok;
        if (ctx->dense_ok) *ctx->maps = *leader->maps;
    }
    if (ctx->dense_ok) {
        std::vector<CUtensorMap>& m = *ctx->maps;
        ctx->dense_ok = make_map(&m[MAP_XN], ws + ctx->r.dxn, kDenseMaxRows, d, 128) && make_map(&m[MAP_ATT], ws + ctx->r.datt, kDenseMaxRows, nq, 128) &&
                        make_map(&m[MAP_ACT], ws + ctx->r.dact, kDenseMaxRows, f, 128) &&
                        make_map(&m[MAP_K], P.kcache, (uint64_t)cfg->n_layers * cfg->n_kv_heads * cfg->max_seq, hd, 128) &&
                        make_map(&m[MAP_V], P.vcache, (uint64_t)cfg->n_layers * cfg->n_kv_heads * cfg->max_seq, hd, 128);
        if (!leader) ctx->dense_ok = ctx->dense_ok && make_map(&m[MAP_LM], ws + ctx->r.dlm, cfg->vocab, d, 128);
        for (int l = 0; l < cfg->n_layers && ctx->dense_ok && !leader; ++l) {
            uint8_t* lb = ws + ctx->r.dw + (size_t)l * ctx->r.layer_stride;
            const size_t o1 = (size_t)nqkv * d * 2, o2 = o1 + (size_t)d * nq * 2, o3 = o2 + (size_t)2 * f * d * 2;
            for (int bn = 128; bn <= 256 && ctx->dense_ok; bn *= 2)
                ctx->dense_ok = make_map(&m[map_at(l, 0, bn)], lb, nqkv, d, bn / 2) && make_map(&m[map_at(l, 1, bn)], lb + o1, d, nq, bn / 2) &&
                                make_map(&m[map_at(l, 2, bn)], lb + o2, 2 * (uint64_t)f, d, bn / 2) && make_map(&m[map_at(l, 3, bn)], lb + o3, d, f, bn / 2);
        }
    }
    ctx->logits_src = P.logits;
    ctx->weights_loaded = leader != nullptr;
    *out = ctx;
    return SDV_OK;
}
}  // namespace

extern "C" {

int sdv_create(const sdv_config* cfg, void* dev_workspace, size_t bytes, void* cuda_stream, sdv_ctx** out) {
    return create_context(cfg, dev_workspace, bytes, (cudaStream_t)cuda_stream, nullptr, out);
}

size_t sdv_follower_workspace_bytes(const sdv_config* cfg) {
    if (!config_ok(cfg)) return 0;
    return carve(cfg, false).total;
}

int sdv_create_follower(sdv_ctx* leader, void* dev_workspace, size_t bytes, sdv_ctx** out) {
    if (out) *out = nullptr;
    if (!leader || leader->leader) return SDV_EINVAL;  // followers follow a context that owns its weights
    if (!leader->weights_loaded) return SDV_ESTATE;
    return create_context(&leader->cfg, dev_workspace, bytes, leader->stream, leader, out);
}

int sdv_destroy(sdv_ctx* ctx) {
    if (!ctx) return SDV_EINVAL;
    cudaStreamSynchronize(ctx->stream);
    if (ctx->pinned) cudaFreeHost(ctx->pinned);
    cudaEventDestroy(ctx->ev0);
    cudaEventDestroy(ctx->ev1);
    delete ctx->maps;
    if (ctx->run_ev) {
        for (cudaEvent_t ev : *ctx->run_ev) cudaEventDestroy(ev);
        delete ctx->run_ev;
    }
    delete ctx;
    return SDV_OK;
}

int sdv_load_weights(sdv_ctx* ctx, const sdv_weights* w) {
    if (!ctx || !w || !w->emb || !w->final_norm || !w->layers) return SDV_EINVAL;
    if (ctx->leader) return SDV_ESTATE;
    const sdv_config& c = ctx->cfg;
    if (!c.tied_lm_head && !w->lm_head) return SDV_EINVAL;
    const size_t d = c.d_model, f = c.d_ffn, hd = c.head_dim, V = c.vocab;
    const size_t nq = c.n_q_heads * hd, nkv = c.n_kv_heads * hd, nqkv = nq + 2 * nkv;
    uint8_t* ws = ctx->ws;
    uint16_t* stg = (uint16_t*)(ws + ctx->r.staging);
    float* norm_w = (float*)(ws + ctx->r.norm_w);
    float* bias = (float*)(ws + ctx->r.bias);
    cudaStream_t s = ctx->stream;
    for (int l = 0; l < c.n_layers; ++l) {
        const sdv_layer_weights& L = w->layers[l];
        if (!L.wq || !L.wk || !L.wv || !L.wo || !L.wg || !L.wu || !L.wd || !L.norm1 || !L.norm2) return SDV_EINVAL;
        if (c.qkv_bias && (!L.bq || !L.bk || !L.bv)) return SDV_EINVAL;
        uint8_t* lbase = ws + ctx->r.wlayers + (size_t)l * ctx->r.layer_stride;
        int rc;
        // q | k | v stacked
        CK(cudaMemcpyAsync(stg, L.wq, nq * d * 2, cudaMemcpyDefault, s));
        CK(cudaMemcpyAsync(stg + nq * d, L.wk, nkv * d * 2, cudaMemcpyDefault, s));
        CK(cudaMemcpyAsync(stg + (nq + nkv) * d, L.wv, nkv * d * 2, cudaMemcpyDefault, s));
        rc = pack_op(ctx, ctx->P.op[OP_QKV], lbase + ctx->P.op[OP_QKV].w_off, stg, (int)nq, stg + nq * d, (int)nkv,
                     stg + (nq + nkv) * d, (int)d, 2, 0, ctx->P.op[OP_QKV].T, 0);
        if (rc) return rc;
        // row-major copies for the dense prefill path: q|k|v, o, gate|up (interleaved by 64), down
        uint16_t* dbase = (uint16_t*)(ws + ctx->r.dw + (size_t)l * ctx->r.layer_stride);
        CK(cudaMemcpyAsync(dbase, stg, nqkv * d * 2, cudaMemcpyDeviceToDevice, s));
        CK(cudaStreamSynchronize(s));
        // o
        CK(cudaMemcpyAsync(stg, L.wo, d * nq * 2, cudaMemcpyDefault, s));
        rc = pack_op(ctx, ctx->P.op[OP_O], lbase + ctx->P.op[OP_O].w_off, stg, (int)d, nullptr, 0, nullptr, (int)nq, 0, 0,
                     ctx->P.op[OP_O].T, 0);
        if (rc) return rc;
        CK(cudaMemcpyAsync(dbase + nqkv * d, stg, d * nq * 2, cudaMemcpyDeviceToDevice, s));
        CK(cudaStreamSynchronize(s));
        // gate | up, interleaved 8 + 8 rows per tile
        CK(cudaMemcpyAsync(stg, L.wg, f * d * 2, cudaMemcpyDefault, s));
        CK(cudaMemcpyAsync(stg + f * d, L.wu, f * d * 2, cudaMemcpyDefault, s));
        rc = pack_op(ctx, ctx->P.op[OP_GU], lbase + ctx->P.op[OP_GU].w_off, stg, (int)f, stg + f * d, (int)f, nullptr,
                     (int)d, 1, 0, ctx->P.op[OP_GU].T, 0);
        if (rc) return rc;
        dense_copy_weights_kernel<<<148 * 8, 256, 0, s>>>(dbase + nqkv * d + d * nq, stg, stg + f * d, (int)(2 * f), (int)d, 1);
        ctx->launches++;
        CK(cudaGetLastError());
        CK(cudaStreamSynchronize(s));
        // down
        CK(cudaMemcpyAsync(stg, L.wd, d * f * 2, cudaMemcpyDefault, s));
        rc = pack_op(ctx, ctx->P.op[OP_DOWN], lbase + ctx->P.op[OP_DOWN].w_off, stg, (int)d, nullptr, 0, nullptr, (int)f,
                     0, 0, ctx->P.op[OP_DOWN].T, 0);
        if (rc) return rc;
        CK(cudaMemcpyAsync(dbase + nqkv * d + d * nq + 2 * f * d, stg, d * f * 2, cudaMemcpyDeviceToDevice, s));
        CK(cudaStreamSynchronize(s));
        CK(cudaMemcpyAsync(norm_w + ((size_t)l * 2 + 0) * d, L.norm1, d * 4, cudaMemcpyDefault, s));
        CK(cudaMemcpyAsync(norm_w + ((size_t)l * 2 + 1) * d, L.norm2, d * 4, cudaMemcpyDefault, s));
        if (c.qkv_bias) {
            CK(cudaMemcpyAsync(bias + (size_t)l * nqkv, L.bq, nq * 4, cudaMemcpyDefault, s));
            CK(cudaMemcpyAsync(bias + (size_t)l * nqkv + nq, L.bk, nkv * 4, cudaMemcpyDefault, s));
            CK(cudaMemcpyAsync(bias + (size_t)l * nqkv + nq + nkv, L.bv, nkv * 4, cudaMemcpyDefault, s));
        }
    }
    CK(cudaMemcpyAsync(norm_w + (size_t)c.n_layers * 2 * d, w->final_norm, d * 4, cudaMemcpyDefault, s));
    CK(cudaMemcpyAsync(ws + ctx->r.emb, w->emb, V * d * 2, cudaMemcpyDefault, s));
    if (!c.tied_lm_head) CK(cudaMemcpyAsync(ws + ctx->r.dlm, w->lm_head, V * d * 2, cudaMemcpyDefault, s));
    // LM head: packed from row blocks that fit the staging area
    {
        const uint16_t* src = c.tied_lm_head ? w->emb : w->lm_head;
        const OpDesc& o = ctx->P.op[OP_LM];
        const size_t tiles_per = ctx->r.staging_bytes / (16 * d * 2);
        if (tiles_per < 1) return SDV_ENOMEM;
        for (size_t t0 = 0; t0 < (size_t)o.T; t0 += tiles_per) {
            const size_t t1 = (t0 + tiles_per < (size_t)o.T) ? t0 + tiles_per : (size_t)o.T;
            const size_t rows = (t1 - t0) * 16;
            CK(cudaMemcpyAsync(stg, src + t0 * 16 * d, rows * d * 2, cudaMemcpyDefault, s));
            int rc = pack_op(ctx, o, ws + ctx->r.wlm, stg, (int)rows, nullptr, 0, nullptr, (int)d, 0, (int)t0, (int)t1,
                             (int)(t0 * 16));
            if (rc) return rc;
            CK(cudaStreamSynchronize(s));
        }
    }
    CK(cudaStreamSynchronize(s));
    ctx->weights_loaded = true;
    return SDV_OK;
}

int sdv_set_parity_mode(sdv_ctx* ctx, int on) {
    if (!ctx) return SDV_EINVAL;
    ctx->parity = on ? 1 : 0;
    return SDV_OK;
}

}  // extern "C"

namespace {
constexpr int kDenseMinRows = 16;  // fewer rows take the small-row kernel
// End of a prefill call: the context covers everything prefilled so far; behind the request's last token (whose
// candidates are those of `row`) the greedy token becomes the pending one and the calibration looks its anchors up.
int finish_prefill(sdv_ctx* ctx, bool is_last, int row) {
    int* hist = (int*)(ctx->ws + ctx->r.hist);
    ctx->n_ctx = ctx->hist_len;
    set_state_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, ctx->kv_len, ctx->hist_len, ctx->n_ctx, 0, hist, ctx->pinned);
    ctx->launches++;
    CK(cudaGetLastError());
    if (!is_last) return SDV_OK;
    // greedy token of the last context row: appended to the history as the pending token T
    prefill_final_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, hist, ctx->P.cand_val, ctx->P.cand_idx, ctx->G, row);
    ctx->launches++;
    CK(cudaGetLastError());
    ctx->hist_len += 1;
    ctx->prefill_done = true;
    if (ctx->calib_b > 0) {
        // "Search": where each sampled successor occurs in the request
        const int total = ctx->n_ctx * ctx->calib_b;
        anchor_search_kernel<<<(total + 255) / 256, 256, 0, ctx->stream>>>(hist, ctx->n_ctx, ctx->calib_b, (const int*)(ctx->ws + ctx->r.succ),
                                                                           (int*)(ctx->ws + ctx->r.occ));
        ctx->launches++;
        CK(cudaGetLastError());
        ctx->calibrated = true;
    }
    return SDV_OK;
}
}  // namespace

extern "C" {

int sdv_prefill_chunk(sdv_ctx* ctx, const int32_t* host_tokens, int n, int is_last) {
    if (!ctx || !host_tokens || n < 1) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->weights_loaded || ctx->prefill_done) return SDV_ESTATE;
    const sdv_config& c = ctx->cfg;
    if (ctx->kv_len + n + 1 + c.k_max + 1 > c.max_seq) return SDV_ECAPACITY;
    for (int i = 0; i < n; ++i)
        if (host_tokens[i] < 0 || host_tokens[i] >= c.vocab) return SDV_EINVAL;
    int* hist = (int*)(ctx->ws + ctx->r.hist);
    CK(cudaMemcpyAsync(hist + ctx->hist_len, host_tokens, (size_t)n * 4, cudaMemcpyDefault, ctx->stream));
    // rows per launch of the small-row kernel
    int tile = 24;
    {
        // wide models: fewer rows per launch so that the token operand leaves room for the weight ring
        FwdParams probe = ctx->P;
        while (tile > 8 && (!apply_plan(probe, tile, false) || probe.nstage < 4)) tile -= 8;
    }
    const int n_ph = 1 + kPhasesPerLayer * c.n_layers;
    int done = 0;
    while (done < n) {
        // sub-chunks of up to kDenseMaxRows rows, evenly cut, go through the dense path (tokens on the tensor cores' M
        // side, every weight streamed once); a handful of rows takes the small-row kernel
        const int left = n - done;
        if (ctx->dense_ok && left >= kDenseMinRows) {
            const int parts = (left + kDenseMaxRows - 1) / kDenseMaxRows, rows = (left + parts - 1) / parts;
            int rc = dense_prefill_rows(ctx, rows, ctx->kv_len, ctx->calib_b > 0 ? (int*)(ctx->ws + ctx->r.succ) + (size_t)ctx->kv_len * ctx->calib_b : nullptr);
            if (rc) return rc;
            ctx->kv_len += rows;
            ctx->hist_len += rows;
            done += rows;
            if (done == n) {
                if (is_last) {
                    // the request's last token gives the first generated one: the LM head over its row alone
                    rc = launch_forward(ctx, 1, ctx->kv_len, 1, n_ph, n_ph + 1, false);
                    if (rc) return rc;
                }
                rc = finish_prefill(ctx, is_last != 0, 0);
                if (rc) return rc;
            }
            continue;
        }
        const int rows = (n - done < tile) ? n - done : tile;
        const bool last_tile = is_last && (done + rows == n);
        const bool calib = ctx->calib_b > 0;
        int rc = launch_forward(ctx, rows, ctx->kv_len, 1, 0, (last_tile || calib) ? n_ph + 1 : n_ph, false, calib);
        if (rc) return rc;
        if (calib) {
            // "Sample": the best successors of every row of this tile, from the logits the LM head just stored
            top_successors_kernel<<<rows, 1024, 0, ctx->stream>>>(ctx->P.logits, c.vocab, ctx->calib_b,
                                                               (int*)(ctx->ws + ctx->r.succ) + (size_t)ctx->kv_len * ctx->calib_b);
            ctx->launches++;
            CK(cudaGetLastError());
        }
        ctx->kv_len += rows;
        ctx->hist_len += rows;
        done += rows;
        if (done == n) {
            rc = finish_prefill(ctx, last_tile, rows - 1);
            if (rc) return rc;
        }
    }
    return read_state(ctx, true);   // finish_prefill's kernel wrote the error word to the host
}

int sdv_draft(sdv_ctx* ctx, int k, int32_t* host_draft, int* draft_len) {
    if (!ctx || k < 1 || k > ctx->cfg.k_max) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->prefill_done) return SDV_ESTATE;
    int* hist = (int*)(ctx->ws + ctx->r.hist);
    ngram_draft_kernel<<<1, 1024, 0, ctx->stream>>>(ctx->P.state, hist, (const int*)(ctx->ws + ctx->r.db), ctx->cfg.ngram_n,
                                                    ctx->cfg.ngram_min, k, ctx->cfg.search_history, 0,
                                                    host_draft || draft_len ? ctx->pinned : nullptr);
    ctx->launches++;
    CK(cudaGetLastError());
    ctx->draft_pending = true;
    ctx->tree_pending = false;
    ctx->draft_k = k;
    ctx->verified = false;
    if (host_draft || draft_len) {
        int rc = read_state(ctx, true);
        if (rc) return rc;
        const int dl = ctx->pinned[ST_DRAFT_LEN];
        if (draft_len) *draft_len = dl;
        if (host_draft)
            for (int i = 0; i < dl; ++i) host_draft[i] = ctx->pinned[ST_DRAFT + i];
    }
    return SDV_OK;
}

int sdv_verify(sdv_ctx* ctx, const int32_t* host_draft, int draft_len, int32_t* host_y, int* accept_len) {
    if (!ctx) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->prefill_done || !ctx->weights_loaded) return SDV_ESTATE;
    const sdv_config& c = ctx->cfg;
    int rows;
    if (host_draft) {
        if (draft_len < 0 || draft_len > c.k_max) return SDV_EINVAL;
        for (int i = 0; i < draft_len; ++i)
            if (host_draft[i] < 0 || host_draft[i] >= c.vocab) return SDV_EINVAL;
        rows = draft_len + 1;
    } else {
        rows = ctx->draft_pending ? ctx->draft_k + 1 : 1;
    }
    if (ctx->kv_len + rows > c.max_seq) return SDV_ECAPACITY;
    // no draft at all: an empty one goes along, since the device may still hold the one of a verify before
    const bool pass = host_draft || !ctx->draft_pending;
    DraftArg a;
    if (pass) fill_draft_arg(a, host_draft, host_draft ? draft_len : 0);
    const bool tree = !host_draft && ctx->tree_pending, fetch = host_y || accept_len;
    int rc = launch_forward(ctx, rows, ctx->kv_len, 0, 0, 2 + kPhasesPerLayer * c.n_layers, true, false, tree, nullptr, false, nullptr,
                            pass ? &a : nullptr);
    if (rc) return rc;
    accept_kernel<<<1, 32 * rows, 0, ctx->stream>>>(ctx->P.state, ctx->P.cand_val, ctx->P.cand_idx, ctx->G, 0,
                                                    fetch ? ctx->pinned : nullptr);
    ctx->launches++;
    CK(cudaGetLastError());
    if (host_draft && ctx->draft_pending) ctx->draft_k = draft_len;   // it has taken the drafter's place on the device
    ctx->verified = true;
    ctx->tree_verified = tree;
    ctx->last_rows = rows;
    if (fetch) {
        rc = read_state(ctx, true);
        if (rc) return rc;
        const int dl = ctx->pinned[ST_DRAFT_LEN];
        if (accept_len) *accept_len = ctx->pinned[ST_ACCEPT_LEN];
        if (host_y)
            for (int i = 0; i <= dl; ++i) host_y[i] = ctx->pinned[ST_Y + i];
    }
    return SDV_OK;
}

int sdv_verify_batch(sdv_ctx* const* ctxs, int n, int* accept_len) {
    if (!ctxs || n < 1 || n > kMaxBatch) return SDV_EINVAL;
    sdv_ctx* ctx = ctxs[0];  // the launch runs on the first context's scratch buffers and stream
    if (!ctx) return SDV_EINVAL;
    sdv_ctx* owner = ctx->leader ? ctx->leader : ctx;
    BatchPlan bp;
    BatchGatherArg ga;
    memset(&bp, 0, sizeof(bp));
    memset(&ga, 0, sizeof(ga));
    bp.n = ga.n = n;
    int rows = 0, Lmax = 0;
    for (int b = 0; b < n; ++b) {
        sdv_ctx* c = ctxs[b];
        if (!c) return SDV_EINVAL;
        for (int a = 0; a < b; ++a)
            if (ctxs[a] == c) return SDV_EINVAL;
        if ((c->leader ? c->leader : c) != owner || c->stream != ctx->stream) return SDV_EINVAL;
        if (c->poisoned) return SDV_ETIMEOUT;
        if (!c->prefill_done || !c->weights_loaded || c->tree_pending) return SDV_ESTATE;  // chains only
        const int m = c->draft_pending ? c->draft_k + 1 : 1;
        if (c->kv_len + m > c->cfg.max_seq) return SDV_ECAPACITY;
        bp.seq[b].kcache = c->P.kcache;
        bp.seq[b].vcache = c->P.vcache;
        bp.seq[b].r0 = ga.r0[b] = rows;
        bp.seq[b].M = ga.M[b] = m;
        bp.seq[b].L = c->kv_len;
        ga.state[b] = c->P.state;
        if (m > bp.max_rows) bp.max_rows = m;
        if (c->kv_len > Lmax) Lmax = c->kv_len;
        rows += m;
    }
    if (rows > kMaxRows) return SDV_EINVAL;
    int* bstate = (int*)(ctx->ws + ctx->r.bstate);
    batch_gather_kernel<<<1, kMaxRows, 0, ctx->stream>>>(bstate, ga);
    ctx->launches++;
    CK(cudaGetLastError());
    int rc = launch_forward(ctx, rows, Lmax, 0, 0, 2 + kPhasesPerLayer * ctx->cfg.n_layers, true, false, false, &bp);
    if (rc) return rc;
    BatchAcceptArg aa;
    memset(&aa, 0, sizeof(aa));
    for (int b = 0; b < n; ++b) {
        sdv_ctx* c = ctxs[b];
        aa.state[b] = c->P.state;
        aa.host[b] = accept_len ? c->pinned : nullptr;
        aa.r0[b] = bp.seq[b].r0;
        aa.M[b] = bp.seq[b].M;
        c->verified = true;
        c->tree_verified = false;
        c->last_rows = bp.seq[b].M;
        c->logits_src = ctx->P.logits + (size_t)bp.seq[b].r0 * ctx->cfg.vocab;
    }
    accept_batch_kernel<<<n, 32 * bp.max_rows, 0, ctx->stream>>>(aa, ctx->P.cand_val, ctx->P.cand_idx, ctx->G, bstate);
    ctx->launches++;
    CK(cudaGetLastError());
    if (accept_len) {
        for (int b = 0; b < n; ++b) {
            sdv_ctx* c = ctxs[b];
            rc = read_state(c, true);
            if (rc) return rc;
            accept_len[b] = c->pinned[ST_ACCEPT_LEN];
        }
    }
    return SDV_OK;
}

int sdv_get_verified(sdv_ctx* ctx, int32_t* host_y, int* accept_len) {
    if (!ctx) return SDV_EINVAL;
    if (!ctx->verified) return SDV_ESTATE;
    int drafts = 0;
    int rc = verified_drafts(ctx, &drafts);
    if (rc) return rc;
    if (accept_len) *accept_len = ctx->pinned[ST_ACCEPT_LEN];
    if (host_y)
        for (int i = 0; i <= drafts; ++i) host_y[i] = ctx->pinned[ST_Y + i];
    return SDV_OK;
}

int sdv_set_database(sdv_ctx* ctx, const int32_t* host_tokens, int n) {
    if (!ctx || n < 0 || n > ctx->cfg.max_seq || (n && !host_tokens)) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    for (int i = 0; i < n; ++i)
        if (host_tokens[i] < 0 || host_tokens[i] >= ctx->cfg.vocab) return SDV_EINVAL;
    if (n) CK(cudaMemcpyAsync(ctx->ws + ctx->r.db, host_tokens, (size_t)n * 4, cudaMemcpyDefault, ctx->stream));
    set_word_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, ST_DB_LEN, n);
    ctx->launches++;
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(ctx->stream));  // the caller's buffer may go away
    return SDV_OK;
}

int sdv_extend_draft(sdv_ctx* ctx, int max_total, int32_t* host_draft, int* draft_len) {
    if (!ctx || max_total < 1 || max_total > ctx->cfg.k_max) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->prefill_done || !ctx->draft_pending) return SDV_ESTATE;
    extend_draft_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, max_total, 0);
    ctx->launches++;
    CK(cudaGetLastError());
    // rows of the next verify: the exact draft length when the caller reads it, else the bound
    if (ctx->draft_k < max_total) ctx->draft_k = max_total;
    if (host_draft || draft_len) {
        int rc = read_state(ctx);
        if (rc) return rc;
        const int dl = ctx->pinned[ST_DRAFT_LEN];
        ctx->draft_k = dl;
        if (draft_len) *draft_len = dl;
        if (host_draft)
            for (int i = 0; i < dl; ++i) host_draft[i] = ctx->pinned[ST_DRAFT + i];
    }
    return SDV_OK;
}

int sdv_extension_update(sdv_ctx* ctx, int max_life, int32_t* host_segment, int* segment_len, int* lifetime) {
    if (!ctx || max_life < 1) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->verified) return SDV_ESTATE;
    extension_update_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, max_life);
    ctx->launches++;
    CK(cudaGetLastError());
    if (host_segment || segment_len || lifetime) {
        int rc = read_state(ctx);
        if (rc) return rc;
        const int sl = ctx->pinned[ST_SEG_LEN];
        if (segment_len) *segment_len = sl;
        if (lifetime) *lifetime = ctx->pinned[ST_SEG_LIFE];
        if (host_segment)
            for (int i = 0; i < sl; ++i) host_segment[i] = ctx->pinned[ST_SEG + i];
    }
    return SDV_OK;
}

int sdv_step(sdv_ctx* ctx, const int32_t* host_draft, int draft_len, int k_next, int32_t* host_emitted, int* n_emitted,
             int32_t* host_next_draft, int* next_draft_len, int* kv_len) {
    if (!ctx || k_next < 0 || k_next > ctx->cfg.k_max) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->prefill_done || !ctx->weights_loaded) return SDV_ESTATE;
    const sdv_config& c = ctx->cfg;
    int rows;
    if (host_draft) {
        if (draft_len < 0 || draft_len > c.k_max) return SDV_EINVAL;
        for (int i = 0; i < draft_len; ++i)
            if (host_draft[i] < 0 || host_draft[i] >= c.vocab) return SDV_EINVAL;
        rows = draft_len + 1;
    } else {
        if (ctx->tree_pending) return SDV_ESTATE;  // chains only
        rows = ctx->draft_pending ? ctx->draft_k + 1 : 1;
    }
    if (ctx->kv_len + rows > c.max_seq || ctx->hist_len + rows > c.max_seq + 64) return SDV_ECAPACITY;
    int* state = ctx->P.state;
    int* hist = (int*)(ctx->ws + ctx->r.hist);
    const bool pass = host_draft || !ctx->draft_pending;   // as in sdv_verify
    DraftArg a;
    if (pass) fill_draft_arg(a, host_draft, host_draft ? draft_len : 0);
    int rc = launch_forward(ctx, rows, ctx->kv_len, 0, 0, 2 + kPhasesPerLayer * c.n_layers, true, false, false, nullptr, false, nullptr,
                            pass ? &a : nullptr);
    if (rc) return rc;
    step_tail_kernel<<<1, 1024, 0, ctx->stream>>>(state, hist, (const int*)(ctx->ws + ctx->r.db), ctx->P.cand_val, ctx->P.cand_idx,
                                                  ctx->G, c.ngram_n, c.ngram_min, k_next, c.search_history, 0, 0, k_next > 0 ? 1 : 0, 0, ctx->pinned, 0, 0);
    ctx->launches++;
    CK(cudaGetLastError());
    ctx->last_rows = rows;
    ctx->verified = false;
    ctx->tree_pending = false;
    ctx->tree_verified = false;
    ctx->draft_pending = k_next > 0;
    ctx->draft_k = k_next;
    rc = read_state(ctx, true);  // the tail kernel wrote the state block to the host: emitted tokens, lengths and the next draft
    if (rc) return rc;
    const int n = ctx->pinned[ST_N_EMITTED];
    ctx->kv_len = ctx->pinned[ST_KV_LEN];
    ctx->hist_len = ctx->pinned[ST_HIST_LEN];
    if (n_emitted) *n_emitted = n;
    if (kv_len) *kv_len = ctx->kv_len;
    if (host_emitted)
        for (int i = 0; i < n; ++i) host_emitted[i] = ctx->pinned[ST_EMITTED + i];
    const int dl = k_next > 0 ? ctx->pinned[ST_DRAFT_LEN] : 0;
    if (next_draft_len) *next_draft_len = dl;
    if (host_next_draft)
        for (int i = 0; i < dl; ++i) host_next_draft[i] = ctx->pinned[ST_DRAFT + i];
    return SDV_OK;
}

int sdv_decode_steps(sdv_ctx* ctx, int k, int n_steps, int max_tokens, int ext_max_total, int ext_max_life, int32_t* host_tokens,
                     int* n_tokens, int* kv_len) {
    if (!ctx || k < 1 || k > ctx->cfg.k_max || n_steps < 1 || n_steps > 4096) return SDV_EINVAL;
    if (ext_max_total < 0 || ext_max_total > ctx->cfg.k_max || (ext_max_total > 0 && (ext_max_total < k || ext_max_life < 1)))
        return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->prefill_done || !ctx->weights_loaded) return SDV_ESTATE;
    const sdv_config& c = ctx->cfg;
    const int rows = (ext_max_total > 0 ? ext_max_total : k) + 1;
    // every step may write `rows` KV rows beyond the length it starts from and emit up to `rows` tokens
    if ((long long)ctx->kv_len + (long long)n_steps * rows > c.max_seq) return SDV_ECAPACITY;
    if ((long long)ctx->hist_len + (long long)n_steps * rows > c.max_seq + 64) return SDV_ECAPACITY;
    if (!ctx->run_ev) ctx->run_ev = new (std::nothrow) std::vector<cudaEvent_t>();
    if (!ctx->run_ev) return SDV_ENOMEM;
    while (ctx->run_ev->size() < 2 * (size_t)n_steps) {
        cudaEvent_t ev;
        CK(cudaEventCreate(&ev));
        ctx->run_ev->push_back(ev);
    }
    int* state = ctx->P.state;
    int* hist = (int*)(ctx->ws + ctx->r.hist);
    const int hist_before = ctx->hist_len;
    fill_i32_kernel<<<1, 32, 0, ctx->stream>>>(state + ST_BUDGET, max_tokens > 0 ? max_tokens : -1, 1);
    const int* db = (const int*)(ctx->ws + ctx->r.db);
    ngram_draft_kernel<<<1, 1024, 0, ctx->stream>>>(state, hist, db, c.ngram_n, c.ngram_min, k, c.search_history, 1, nullptr);
    if (ext_max_total > 0) extend_draft_kernel<<<1, 32, 0, ctx->stream>>>(state, ext_max_total, 1);
    ctx->launches += ext_max_total > 0 ? 3 : 2;
    const int all_phases = 2 + kPhasesPerLayer * c.n_layers, room = kPinnedBytes / 4 - ST_WORDS;
    for (int i = 0; i < n_steps; ++i) {
        // the kernel reads the KV length from the state block; the host's value (a lower bound) only shapes the attention split
        int rc = launch_forward(ctx, rows, ctx->kv_len, 0, 0, all_phases, true, false, false, nullptr, true,
                                ctx->run_ev->data() + 2 * i);
        if (rc) return rc;
        // accept, commit and the next step's draft in one launch
        step_tail_kernel<<<1, 1024, 0, ctx->stream>>>(state, hist, db, ctx->P.cand_val, ctx->P.cand_idx, ctx->G, c.ngram_n,
                                                      c.ngram_min, k, c.search_history, ext_max_total, ext_max_life,
                                                      i + 1 < n_steps ? 1 : 0, 1, i + 1 < n_steps ? nullptr : ctx->pinned, hist_before,
                                                      i + 1 < n_steps ? 0 : room);
        ctx->launches++;
    }
    CK(cudaGetLastError());
    ctx->run_steps = n_steps;
    ctx->verified = false;
    ctx->draft_pending = false;
    ctx->tree_pending = false;
    ctx->tree_verified = false;
    int rc = read_state(ctx, true);   // written by the last tail kernel, tokens too
    if (rc) return rc;
    ctx->kv_len = ctx->pinned[ST_KV_LEN];
    ctx->hist_len = ctx->pinned[ST_HIST_LEN];
    const int n = ctx->hist_len - hist_before;
    if (n_tokens) *n_tokens = n;
    if (kv_len) *kv_len = ctx->kv_len;
    if (host_tokens && n > 0 && n <= room) {
        memcpy(host_tokens, ctx->pinned + ST_WORDS, (size_t)n * 4);
    } else if (host_tokens && n > 0) {
        CK(cudaMemcpyAsync(host_tokens, hist + hist_before, (size_t)n * 4, cudaMemcpyDeviceToHost, ctx->stream));
        CK(cudaStreamSynchronize(ctx->stream));
    }
    return SDV_OK;
}

int sdv_run_kernel_ms(sdv_ctx* ctx, float* host_ms, int n) {
    if (!ctx || !host_ms || n < 1) return SDV_EINVAL;
    if (!ctx->run_ev || n > ctx->run_steps) return SDV_ESTATE;
    CK(cudaStreamSynchronize(ctx->stream));
    for (int i = 0; i < n; ++i) CK(cudaEventElapsedTime(&host_ms[i], (*ctx->run_ev)[2 * i], (*ctx->run_ev)[2 * i + 1]));
    return SDV_OK;
}

int sdv_set_calibration(sdv_ctx* ctx, int top_b) {
    if (!ctx || top_b < 0 || top_b > SDV_CALIB_MAX) return SDV_EINVAL;
    if (ctx->kv_len > 0 || ctx->prefill_done) return SDV_ESTATE;  // the tables are filled while the context is prefilled
    ctx->calib_b = top_b;
    ctx->calibrated = false;
    return SDV_OK;
}

int sdv_get_calibration(sdv_ctx* ctx, int32_t* host_succ, int32_t* host_occ, int n_positions) {
    if (!ctx || n_positions < 1 || (!host_succ && !host_occ)) return SDV_EINVAL;
    if (!ctx->calibrated) return SDV_ESTATE;
    if (n_positions > ctx->n_ctx) return SDV_EINVAL;
    const size_t bytes = (size_t)n_positions * ctx->calib_b * 4;
    if (host_succ) CK(cudaMemcpyAsync(host_succ, ctx->ws + ctx->r.succ, bytes, cudaMemcpyDeviceToHost, ctx->stream));
    if (host_occ) CK(cudaMemcpyAsync(host_occ, ctx->ws + ctx->r.occ, bytes, cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    return SDV_OK;
}

int sdv_draft_tree(sdv_ctx* ctx, int k, int max_nodes, int32_t* host_tokens, int32_t* host_parent, int* n_nodes) {
    if (!ctx || k < 0 || k > ctx->cfg.k_max || max_nodes < 1 || max_nodes > ctx->cfg.k_max) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->prefill_done) return SDV_ESTATE;
    int* hist = (int*)(ctx->ws + ctx->r.hist);
    if (k > 0) {
        ngram_draft_kernel<<<1, 1024, 0, ctx->stream>>>(ctx->P.state, hist, (const int*)(ctx->ws + ctx->r.db), ctx->cfg.ngram_n,
                                                        ctx->cfg.ngram_min, k, ctx->cfg.search_history, 0, nullptr);
    } else {
        DraftArg none;
        fill_draft_arg(none, nullptr, 0);
        set_draft_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, none);
    }
    tree_draft_kernel<<<1, 1024, 0, ctx->stream>>>(ctx->P.state, hist, (const int*)(ctx->ws + ctx->r.succ),
                                                   (const int*)(ctx->ws + ctx->r.occ), ctx->calibrated ? ctx->calib_b : 0, max_nodes,
                                                   host_tokens || host_parent || n_nodes ? ctx->pinned : nullptr);
    ctx->launches += 2;
    CK(cudaGetLastError());
    ctx->draft_pending = true;
    ctx->tree_pending = true;
    ctx->draft_k = max_nodes;   // rows of the next verify: the bound, or the exact count when the caller reads it
    ctx->verified = false;
    if (host_tokens || host_parent || n_nodes) {
        int rc = read_state(ctx, true);
        if (rc) return rc;
        const int n = ctx->pinned[ST_DRAFT_LEN];
        ctx->draft_k = n;
        if (n_nodes) *n_nodes = n;
        for (int i = 0; i < n; ++i) {
            if (host_tokens) host_tokens[i] = ctx->pinned[ST_DRAFT + i];
            if (host_parent) host_parent[i] = ctx->pinned[ST_PARENT + 1 + i];
        }
    }
    return SDV_OK;
}

int sdv_verify_tree(sdv_ctx* ctx, const int32_t* host_tokens, const int32_t* host_parent, int n_nodes, int32_t* host_y,
                    int32_t* host_path, int* path_len) {
    if (!ctx) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->prefill_done || !ctx->weights_loaded) return SDV_ESTATE;
    const sdv_config& c = ctx->cfg;
    int rows;
    if (host_tokens) {
        if (!host_parent || n_nodes < 0 || n_nodes > c.k_max) return SDV_EINVAL;
        for (int i = 0; i < n_nodes; ++i) {
            if (host_tokens[i] < 0 || host_tokens[i] >= c.vocab) return SDV_EINVAL;
            if (host_parent[i] < 0 || host_parent[i] > i) return SDV_EINVAL;  // node i + 1 continues an earlier row
        }
        rows = n_nodes + 1;
    } else {
        if (!ctx->tree_pending) return SDV_ESTATE;
        rows = ctx->draft_k + 1;
    }
    if (ctx->kv_len + rows > c.max_seq) return SDV_ECAPACITY;
    if (host_tokens) {
        DraftArg t, p;
        fill_draft_arg(t, host_tokens, n_nodes);
        fill_draft_arg(p, host_parent, n_nodes);
        set_tree_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, t, p);
        ctx->launches++;
        CK(cudaGetLastError());
    }
    int rc = launch_forward(ctx, rows, ctx->kv_len, 0, 0, 2 + kPhasesPerLayer * c.n_layers, true, false, true);
    if (rc) return rc;
    const bool fetch = host_y || host_path || path_len;
    accept_kernel<<<1, 32 * rows, 0, ctx->stream>>>(ctx->P.state, ctx->P.cand_val, ctx->P.cand_idx, ctx->G, 0,
                                                    fetch ? ctx->pinned : nullptr);
    ctx->launches++;
    CK(cudaGetLastError());
    ctx->verified = true;
    ctx->tree_verified = true;
    ctx->last_rows = rows;
    if (fetch) {
        rc = read_state(ctx, true);
        if (rc) return rc;
        const int n = ctx->pinned[ST_DRAFT_LEN], a = ctx->pinned[ST_PATH_LEN];
        if (path_len) *path_len = a;
        if (host_path)
            for (int i = 0; i < a; ++i) host_path[i] = ctx->pinned[ST_PATH + i];
        if (host_y)
            for (int i = 0; i <= n; ++i) host_y[i] = ctx->pinned[ST_Y + i];
    }
    return SDV_OK;
}

int sdv_debug_force_commit_tree(sdv_ctx* ctx, const int32_t* host_path, int path_len, int32_t next_token) {
    if (!ctx || path_len < 0 || (path_len && !host_path)) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->verified || !ctx->tree_verified) return SDV_ESTATE;
    if (next_token < 0 || next_token >= ctx->cfg.vocab) return SDV_EINVAL;
    int nodes = 0;
    int rc = verified_drafts(ctx, &nodes);
    if (rc) return rc;
    if (path_len > nodes) return SDV_EINVAL;
    for (int i = 0; i < path_len; ++i)
        if (host_path[i] < 1 || host_path[i] > nodes || (i && host_path[i] <= host_path[i - 1])) return SDV_EINVAL;
    DraftArg p;
    fill_draft_arg(p, host_path, path_len);
    set_path_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, p, next_token);
    ctx->launches++;
    CK(cudaGetLastError());
    return commit_common(ctx, 0, -1, 0, nullptr, nullptr, nullptr);
}

int sdv_commit(sdv_ctx* ctx, int max_emit, int32_t* host_emitted, int* n_emitted, int* kv_len) {
    if (!ctx) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->verified) return SDV_ESTATE;
    return commit_common(ctx, max_emit, -1, 0, host_emitted, n_emitted, kv_len);
}

int sdv_debug_force_commit(sdv_ctx* ctx, int accept_len, int32_t next_token) {
    if (!ctx) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->verified) return SDV_ESTATE;
    if (accept_len < 0 || next_token < 0 || next_token >= ctx->cfg.vocab) return SDV_EINVAL;
    int drafts = 0;
    int rc = verified_drafts(ctx, &drafts);
    if (rc) return rc;
    if (accept_len > drafts) return SDV_EINVAL;
    return commit_common(ctx, 0, accept_len, next_token, nullptr, nullptr, nullptr);
}

int sdv_rollback(sdv_ctx* ctx, int new_kv_len) {
    if (!ctx) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (!ctx->prefill_done) return SDV_ESTATE;
    if (new_kv_len < 1 || new_kv_len > ctx->kv_len) return SDV_EINVAL;
    int* hist = (int*)(ctx->ws + ctx->r.hist);
    ctx->kv_len = new_kv_len;
    ctx->hist_len = new_kv_len + 1;
    set_state_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, ctx->kv_len, ctx->hist_len, ctx->n_ctx, 1, hist, nullptr);
    ctx->launches++;
    CK(cudaGetLastError());
    ctx->verified = false;
    ctx->draft_pending = false;
    ctx->tree_pending = false;
    ctx->tree_verified = false;
    CK(cudaStreamSynchronize(ctx->stream));
    return SDV_OK;
}

int sdv_get_logits(sdv_ctx* ctx, float* host_logits, int rows) {
    if (!ctx || !host_logits || rows < 1 || rows > kMaxRows) return SDV_EINVAL;
    if (!ctx->parity) return SDV_ESTATE;
    CK(cudaMemcpyAsync(host_logits, ctx->logits_src, (size_t)rows * ctx->cfg.vocab * 4, cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    return SDV_OK;
}

int sdv_step_bytes(const sdv_ctx* ctx, int rows, int kv_len, double* weight_bytes, double* kv_bytes) {
    if (!ctx || rows < 1) return SDV_EINVAL;
    const sdv_config& c = ctx->cfg;
    const double hd = c.head_dim, nq = c.n_q_heads * hd, nkv = c.n_kv_heads * hd, d = c.d_model, f = c.d_ffn;
    const double per_layer = (nq + 2 * nkv) * d + d * nq + 3 * d * f;
    if (weight_bytes) *weight_bytes = 2.0 * (c.n_layers * per_layer + (double)c.vocab * d);
    if (kv_bytes) *kv_bytes = (double)c.n_layers * 2.0 * nkv * 2.0 * ((double)kv_len + rows);
    return SDV_OK;
}

int sdv_last_verify_ms(sdv_ctx* ctx, float* ms) {
    if (!ctx || !ms) return SDV_EINVAL;
    if (!ctx->have_verify_time) return SDV_ESTATE;
    CK(cudaEventSynchronize(ctx->ev1));
    CK(cudaEventElapsedTime(ms, ctx->ev0, ctx->ev1));
    return SDV_OK;
}

// ------------------------------------------------------------------------------------------ debug
int sdv_debug_set_history(sdv_ctx* ctx, const int32_t* host_hist, int hist_len, int n_ctx) {
    if (!ctx || !host_hist || hist_len < 1 || n_ctx < 0 || n_ctx > hist_len) return SDV_EINVAL;
    if (hist_len > ctx->cfg.max_seq) return SDV_ECAPACITY;
    int* hist = (int*)(ctx->ws + ctx->r.hist);
    CK(cudaMemcpyAsync(hist, host_hist, (size_t)hist_len * 4, cudaMemcpyDefault, ctx->stream));
    ctx->hist_len = hist_len;
    ctx->kv_len = hist_len - 1;
    ctx->n_ctx = n_ctx;
    set_state_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, ctx->kv_len, ctx->hist_len, ctx->n_ctx, 1, hist, nullptr);
    ctx->launches++;
    CK(cudaGetLastError());
    ctx->prefill_done = true;
    ctx->verified = false;
    ctx->draft_pending = false;
    ctx->tree_pending = false;
    ctx->tree_verified = false;
    CK(cudaStreamSynchronize(ctx->stream));
    return SDV_OK;
}

int sdv_debug_set_draft(sdv_ctx* ctx, const int32_t* host_draft, int draft_len) {
    if (!ctx || draft_len < 0 || draft_len > ctx->cfg.k_max || (draft_len && !host_draft)) return SDV_EINVAL;
    DraftArg a;
    fill_draft_arg(a, host_draft, draft_len);
    set_draft_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, a);
    ctx->launches++;
    CK(cudaGetLastError());
    ctx->draft_pending = true;
    ctx->tree_pending = false;
    ctx->draft_k = draft_len;
    ctx->verified = false;
    return SDV_OK;
}

int sdv_debug_accept(sdv_ctx* ctx, const int32_t* host_draft, int draft_len, const int32_t* host_y, int* accept_len) {
    if (!ctx || !host_y || draft_len < 0 || draft_len > ctx->cfg.k_max) return SDV_EINVAL;
    DraftArg a, y;
    fill_draft_arg(y, host_y, draft_len + 1);
    if (host_draft) {
        // host_draft == NULL: the draft already on the device (draft_len must be its length)
        fill_draft_arg(a, host_draft, draft_len);
        set_draft_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, a);
        ctx->launches++;
    }
    set_y_kernel<<<1, 32, 0, ctx->stream>>>(ctx->P.state, y);
    accept_kernel<<<1, 32 * (draft_len + 1), 0, ctx->stream>>>(ctx->P.state, ctx->P.cand_val, ctx->P.cand_idx, ctx->G, 1, nullptr);
    ctx->launches += 2;
    CK(cudaGetLastError());
    ctx->verified = true;
    ctx->last_rows = draft_len + 1;
    int rc = read_state(ctx);
    if (rc) return rc;
    if (accept_len) *accept_len = ctx->pinned[ST_ACCEPT_LEN];
    return SDV_OK;
}

int sdv_debug_top_successors(sdv_ctx* ctx, const float* host_logits, int rows, int top_b, int32_t* host_out) {
    if (!ctx || !host_logits || !host_out || rows < 1 || rows > kMaxRows || top_b < 1 || top_b > SDV_CALIB_MAX)
        return SDV_EINVAL;
    const size_t V = ctx->cfg.vocab;
    CK(cudaMemcpyAsync(ctx->ws + ctx->r.logits, host_logits, (size_t)rows * V * 4, cudaMemcpyDefault, ctx->stream));
    int* out = (int*)(ctx->ws + ctx->r.xstage);  // scratch of the stand-alone GEMM: at least 32 * d floats
    top_successors_kernel<<<rows, 1024, 0, ctx->stream>>>(ctx->P.logits, (int)V, top_b, out);
    ctx->launches++;
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(host_out, out, (size_t)rows * top_b * 4, cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    return SDV_OK;
}

int sdv_debug_read_kv(sdv_ctx* ctx, int layer, int which, int pos0, int n, float* host_out) {
    if (!ctx || !host_out || layer < 0 || layer >= ctx->cfg.n_layers || pos0 < 0 || n < 1 ||
        pos0 + n > ctx->cfg.max_seq)
        return SDV_EINVAL;
    const sdv_config& c = ctx->cfg;
    const size_t hd = c.head_dim;
    std::vector<uint16_t> tmp((size_t)n * hd);
    const uint8_t* base = ctx->ws + (which ? ctx->r.vcache : ctx->r.kcache);
    for (int a = 0; a < c.n_kv_heads; ++a) {
        const size_t off = (((size_t)layer * c.n_kv_heads + a) * c.max_seq + pos0) * hd * 2;
        CK(cudaMemcpyAsync(tmp.data(), base + off, tmp.size() * 2, cudaMemcpyDeviceToHost, ctx->stream));
        CK(cudaStreamSynchronize(ctx->stream));
        for (size_t i = 0; i < tmp.size(); ++i) {
            const uint32_t u = (uint32_t)tmp[i] << 16;
            memcpy(&host_out[(size_t)a * n * hd + i], &u, 4);
        }
    }
    return SDV_OK;
}

int sdv_debug_read_hidden(sdv_ctx* ctx, int rows, float* host_out) {
    if (!ctx || !host_out || rows < 1 || rows > kMaxRows) return SDV_EINVAL;
    CK(cudaMemcpyAsync(host_out, ctx->ws + ctx->r.h, (size_t)rows * ctx->cfg.d_model * 4, cudaMemcpyDeviceToHost,
                       ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    return SDV_OK;
}

int sdv_debug_gemm(sdv_ctx* ctx, const float* host_x, const uint16_t* host_w, float* host_y, int M, int N, int K,
                   float* dev_ms) {
    if (!ctx || !host_x || !host_w || !host_y) return SDV_EINVAL;
    if (ctx->poisoned) return SDV_ETIMEOUT;
    if (ctx->leader) return SDV_ESTATE;  // no staging areas without weight regions
    if (M < 1 || M > kMaxRows || N < 16 || N % 16 || K < 64 || K % 64) return SDV_EINVAL;
    if ((size_t)K > ctx->r.raw_kmax || (size_t)N * K * 2 > ctx->r.staging_bytes || (size_t)N > ctx->r.staging_bytes / 128)
        return SDV_EINVAL;
    const sdv_config& c = ctx->cfg;
    uint8_t* ws = ctx->ws;
    cudaStream_t s = ctx->stream;
    OpDesc o;
    memset(&o, 0, sizeof(o));
    o.T = N / 16;
    o.K16 = K / 16;
    choose_partition(o, ctx->G, M, false, false);
    fit_pass_width(o);
    CK(cudaMemcpyAsync(ws + ctx->r.staging, host_w, (size_t)N * K * 2, cudaMemcpyDefault, s));
    int rc = pack_op(ctx, o, ws + ctx->r.wraw, (const uint16_t*)(ws + ctx->r.staging), N, nullptr, 0, nullptr, K, 0, 0,
                     o.T, 0);
    if (rc) return rc;
    CK(cudaMemcpyAsync(ws + ctx->r.xstage, host_x, (size_t)M * K * 4, cudaMemcpyDefault, s));
    CK(cudaMemsetAsync(ws + ctx->r.raw_out, 0, (size_t)kMaxRows * N * 4, s));
    const OpDesc saved = ctx->P.op[OP_RAW];
    const int saved_N = ctx->P.raw_N, saved_K = ctx->P.raw_K;
    ctx->P.op[OP_RAW] = o;
    ctx->P.raw_N = N;
    ctx->P.raw_K = K;
    const int ph = 2 + kPhasesPerLayer * c.n_layers;
    rc = launch_forward(ctx, M, 0, 1, ph, ph + 1, true);
    ctx->P.op[OP_RAW] = saved;
    ctx->P.raw_N = saved_N;
    ctx->P.raw_K = saved_K;
    if (rc) return rc;
    CK(cudaMemcpyAsync(host_y, ws + ctx->r.raw_out, (size_t)M * N * 4, cudaMemcpyDeviceToHost, s));
    rc = read_state(ctx);
    if (rc) return rc;
    if (dev_ms) CK(cudaEventElapsedTime(dev_ms, ctx->ev0, ctx->ev1));
    return SDV_OK;
}

int sdv_debug_profile(sdv_ctx* ctx, int on, unsigned long long* host_out, int n_phases) {
    if (!ctx) return SDV_EINVAL;
    if (host_out) {
        if (n_phases < 1 || n_phases > 3 + kPhasesPerLayer * ctx->cfg.n_layers) return SDV_EINVAL;
        CK(cudaMemcpyAsync(host_out, ctx->ws + ctx->r.prof, (size_t)n_phases * ctx->G * kProfWords * 8, cudaMemcpyDeviceToHost,
                           ctx->stream));
        CK(cudaStreamSynchronize(ctx->stream));
    }
    if (on)
        CK(cudaMemsetAsync(ctx->ws + ctx->r.prof, 0,
                           (size_t)(3 + kPhasesPerLayer * ctx->cfg.n_layers) * kMaxGrid * kProfWords * 8, ctx->stream));
    ctx->profile = on ? 1 : 0;
    return ctx->G;
}

// Host-only self-check of the streaming layout: walks every block's share of an operation the way
// the weight streamer and the tensor-core thread do (pass by pass, stage by stage, the addresses the
// shared-memory descriptors generate) and checks that each 16-byte unit of the matrix is met exactly
// once, at the offset the packing function gives.  desc = {T, K16, P_row, P_k, RW, SK, unit, follow};
// gu_desc likewise (only read when follow is set).  Returns 0, or a negative code.
int sdv_debug_layout_check(const int* desc, const int* gu_desc, int G) {
    if (!desc || !gu_desc || G < 1) return SDV_EINVAL;
    OpDesc o, gu;
    memset(&o, 0, sizeof(o));
    memset(&gu, 0, sizeof(gu));
    o.T = desc[0]; o.K16 = desc[1]; o.P_row = desc[2]; o.P_k = desc[3]; o.RW = desc[4]; o.SK = desc[5]; o.unit = desc[6];
    o.follow = desc[7] & 0xff;
    o.slices = desc[7] >> 8;
    gu.T = gu_desc[0]; gu.K16 = gu_desc[1]; gu.P_row = gu_desc[2]; gu.P_k = gu_desc[3]; gu.RW = gu_desc[4]; gu.SK = gu_desc[5];
    gu.unit = gu_desc[6];
    if (o.T < 1 || o.K16 < 1 || o.RW < 1 || o.SK < 1 || o.RW * o.SK * kStepBytes > kStageBytes || o.unit < 1 || o.T % o.unit) return SDV_EINVAL;
    const int slices = o.slices > 1 ? o.slices : 1;
    if (o.K16 % slices || (slices > 1 && o.P_k != 1) || o.RW * slices * o.SK * kStepBytes > kStageBytes) return SDV_EINVAL;
    const size_t units = (size_t)o.T * 16 * o.K16 * 2;  // 16-byte units of the matrix
    std::vector<unsigned char> seen(units, 0);
    for (int cta = 0; cta < G; ++cta) {
        const Part pt = get_part(o, gu, cta, G);
        if (pt.ntiles == 0 || pt.nk == 0) continue;
        for (int i = 0; i < pt.npass; ++i) {
            const int p = pass_index(pt, i), pcount = pass_count(pt, p), pstart = pass_start(pt, p);
            unsigned long long src = pt.off + (unsigned long long)pstart * pt.nk * kStepBytes;  // the streamer's running offset
            if (pcount < 1 || pcount > 16) return -100;
            const int per = pt.nk / slices, v = pcount * slices;   // column steps per slice; row tiles of the pass, slices stacked
            for (int st = 0; st < pt.nst; ++st) {
                const int nks = (pt.SK < per - st * pt.SK) ? pt.SK : per - st * pt.SK;
                const unsigned long long bytes = (unsigned long long)v * nks * kStepBytes;
                if (bytes > (unsigned long long)kStageBytes) return -101;
                const unsigned lbo = 2u * v * 128u, astep = 2u * lbo;
                for (int ks = 0; ks < nks; ++ks)
                    for (int half = 0; half < 2; ++half)
                        for (int r = 0; r < 16 * v; ++r) {
                            const unsigned long long in_slot = (unsigned long long)ks * astep + half * lbo + (r >> 3) * 128 + (r & 7) * 16;
                            if (in_slot + 16 > bytes) return -102;
                            const int slice = r / (16 * pcount), row = (pt.tile0 + pstart) * 16 + r % (16 * pcount);
                            const int k8 = (pt.k0 + slice * per + st * pt.SK + ks) * 2 + half;
                            const unsigned long long want = weight_offset(o, gu, row, k8);
                            if (want != src + in_slot) return -103;
                            const size_t u = want / 16;
                            if (u >= units || seen[u]) return -104;
                            seen[u] = 1;
                        }
                src += bytes;
            }
        }
    }
    for (size_t u = 0; u < units; ++u)
        if (!seen[u]) return -105;
    return 0;
}

// Host-only: the work partition and shared-memory plan a context of this configuration would use
// with G thread blocks and `rows` token rows.  out[op * 8 + {0..7}] = {T, K16, P_row, P_k, RW, SK,
// unit, follow} for the five operations (QKV, O, gate|up, down, LM head), then out[40..45] =
// {NG, NB, ring slots, operand region bytes, total dynamic shared memory, plan ok}.
int sdv_debug_plan(const sdv_config* cfg, int G, int rows, int* out) {
    if (!config_ok(cfg) || !out || G < 1 || G > kMaxGrid || rows < 1 || rows > kMaxRows) return SDV_EINVAL;
    FwdParams P;
    memset(&P, 0, sizeof(P));
    P.d = cfg->d_model;
    P.hd = cfg->head_dim;
    setup_ops(P, cfg, G, true);
    for (int i = 0; i < 5; ++i) {
        const OpDesc& o = P.op[i];
        const int v[8] = {o.T, o.K16, o.P_row, o.P_k, o.RW, o.SK, o.unit, o.follow | (o.slices << 8)};
        for (int j = 0; j < 8; ++j) out[i * 8 + j] = v[j];
    }
    const SmemPlan sp = plan_smem(P, rows, false);
    out[40] = sp.NG; out[41] = sp.NB; out[42] = sp.nstage; out[43] = sp.u_bytes; out[44] = kSmemBudget; out[45] = sp.ok ? 1 : 0;
    return SDV_OK;
}

int sdv_debug_grid(const sdv_config* cfg, int sms, int clusters, int* blocks, int* in_pairs) {
    if (!config_ok(cfg) || sms < 1 || sms > kMaxGrid || !blocks || !in_pairs) return SDV_EINVAL;
    FwdParams P;
    memset(&P, 0, sizeof(P));
    P.d = cfg->d_model;
    P.hd = cfg->head_dim;
    *blocks = setup_grid(P, cfg, sms, [&]() { return clusters; });
    *in_pairs = P.op[OP_DOWN].P_row == 2 ? 1 : 0;
    return SDV_OK;
}

int sdv_debug_context_grid(const sdv_ctx* ctx, int* blocks, int* in_pairs) {
    if (!ctx || !blocks || !in_pairs) return SDV_EINVAL;
    *blocks = ctx->G;
    *in_pairs = ctx->P.op[OP_DOWN].P_row == 2 ? 1 : 0;
    return SDV_OK;
}

int sdv_debug_pair_debt(int mine, int sent) { return mine < 0 || sent < 0 ? SDV_EINVAL : pair_debt(mine, sent); }

int sdv_debug_timeout_probe(sdv_ctx* ctx) {
    if (!ctx) return SDV_EINVAL;
    timeout_probe_kernel<<<1, 1, 0, ctx->stream>>>(ctx->P.state, (const int*)(ctx->ws + ctx->r.never), 5000000ull);
    ctx->launches++;
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(ctx->pinned, ctx->ws + ctx->r.state, ST_WORDS * 4, cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    const int err = ctx->pinned[ST_ERR];
    CK(cudaMemsetAsync(ctx->P.state + ST_ERR, 0, 4, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    return err == 2 ? SDV_ETIMEOUT : SDV_OK;
}

}  // extern "C"

// ------------------------------------------------------------------------------------------
// Stand-alone GEMM without any allocation (see include/sdv.h, sdv_gemm_noalloc): one kernel on the caller's operands
// (small_gemm.cuh), no scratch.
namespace {
constexpr size_t kNaWeightBytes = (size_t)2 << 20;              // N * K * 2 <= 2 MiB
constexpr int kNaMaxK = 4096, kNaMaxN = 4096;
}  // namespace

extern "C" {

int sdv_gemm_noalloc(const float* dev_x, const uint16_t* dev_w, float* dev_y, int M, int N, int K, void* cuda_stream) {
    if (!dev_x || !dev_w || !dev_y) return SDV_EINVAL;
    if (M < 1 || N < 16 || N % 16 || K < 64 || K % 64) return SDV_EINVAL;
    if (M > kMaxRows || N > kNaMaxN || K > kNaMaxK || (size_t)N * K * 2 > kNaWeightBytes) return SDV_ETOOBIG;
    // the kernel reads x and w with 16-byte vector loads
    if ((((uintptr_t)dev_x | (uintptr_t)dev_w) & 15) || ((uintptr_t)dev_y & 3)) return SDV_EINVAL;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return SDV_ECUDA;
    {
        // host memory or another device's memory would fault inside the kernel: refuse it here
        const void* ptrs[3] = {dev_x, dev_w, dev_y};
        for (int i = 0; i < 3; ++i) {
            cudaPointerAttributes at;
            if (cudaPointerGetAttributes(&at, ptrs[i]) != cudaSuccess) {
                cudaGetLastError();
                return SDV_EINVAL;
            }
            if (at.type == cudaMemoryTypeManaged) continue;
            if (at.type != cudaMemoryTypeDevice || at.device != dev) return SDV_EINVAL;
        }
    }
    // blocks that share the K steps of 16 weight rows: doubled while a warp keeps two steps and the grid stays within about two
    // blocks per SM
    const int tiles = N / 16, steps = K / 32;
    int cs = 1;
    while (cs < 8 && steps >= 2 * (cs * 2) * kSmallGemmWarps && tiles * cs * 2 <= 296) cs *= 2;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(tiles * cs);
    cfg.blockDim = dim3(kSmallGemmWarps * 32);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cs > 1 ? 1 : 0;   // a block alone is a cluster of its own
    typedef void (*Kernel)(const float*, const uint16_t*, float*, int, int, int);
    static const Kernel kernels[4] = {small_gemm_kernel<1>, small_gemm_kernel<2>, small_gemm_kernel<3>, small_gemm_kernel<4>};
    static DeviceOnce loaded;
    // the runtime loads a kernel's code when it is first named: all four now, so that no later call makes it take memory
    const cudaError_t named = loaded.run(dev, []() {
        cudaError_t e = cudaSuccess;
        for (int i = 0; i < 4 && e == cudaSuccess; ++i) {
            cudaFuncAttributes fa;
            e = cudaFuncGetAttributes(&fa, (const void*)kernels[i]);
        }
        return e;
    });
    if (named != cudaSuccess) return SDV_ECUDA;
    if (cudaLaunchKernelEx(&cfg, kernels[(M - 1) / 8], dev_x, dev_w, dev_y, M, N, K) != cudaSuccess) return SDV_ECUDA;
    return cudaStreamSynchronize(s) == cudaSuccess ? SDV_OK : SDV_ECUDA;
}

}  // extern "C"
