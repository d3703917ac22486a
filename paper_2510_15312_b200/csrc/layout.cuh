// Shapes, buffer pointers and the static work partition shared by host code and kernels.
//
// Weight streaming layout.  Every linear layer W[N][K] (bf16) is seen as a grid of T = N/16 row
// tiles by K16 = K/16 column steps (one step = the 16 input features of one tensor-core
// instruction).  The grid is split into P_row x P_k rectangular partitions, one per thread
// block.  A block walks its partition in passes of at most RW row tiles (RW <= 16: one pass is
// one or two 128-row accumulators in tensor memory, rows past the pass are don't-care) and, inside a
// pass, in stages of at most SK column steps (RW * SK <= 64, i.e. <= 32 KB).  A stage is stored
// as the shared-memory image the tensor core reads: column step by column step, the two
// 8-column halves of a step one after the other, each a run of 8-row x 16-byte core matrices
//     [step][half][8-row group][row][8 bf16]
// with no padding.  Stages follow each other pass by pass, so every stage is one contiguous
// bulk copy and a block's whole share of an operation is one contiguous byte range.
//
// A share of few row tiles would leave most of a 128-row instruction empty.  Such an operation is cut into K slices
// that are stacked as rows: with `slices` = 8 the 16 rows of one tile and eighths of their columns fill the 128 rows, the token
// operand is stacked the same way (eight times the token rows), and only the blocks on the diagonal of the product
// are wanted (slice s of the rows against slice s of the tokens); they are added up in the epilogue.  A column step
// of the stage then holds `slices` real column steps, one per slice.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace sdv {

constexpr int kWorkerWarps = 10;                       // every warp but the tensor-core warp and the weight streamer
constexpr int kWorkerThreads = kWorkerWarps * 32;      // 320
constexpr int kThreads = kWorkerThreads + 64;          // 384 with those two
constexpr int kBuilderWarps = kWorkerWarps;            // the workers build the token operand of a GEMM
constexpr int kEpilogueWarps = 8;                      // warps 0..7 read the accumulators: warp w lanes 32(w%4)..+31 of accumulator w/4
constexpr int kMmaWarp = 10;                           // one thread of it issues the tensor-core instructions
constexpr int kProducerWarp = 11;
constexpr int kStepBytes = 512;                        // one row tile x one column step: 16 x 16 bf16
constexpr int kStageBytes = 32768;                     // ring slot
constexpr int kMaxStages = 8;                          // ring slots at most
constexpr int kMaxRows = 32;                           // token rows a buffer is sized for
constexpr int kMaxGrid = 256;                          // thread blocks at most: per-block candidate arrays are sized for them
constexpr int kMaxBatch = 8;                           // sequences one batched verify step takes at most
constexpr int kMaxSplits = 40;                         // key ranges per head at most
constexpr int kSmemBudget = 232448;                    // 227 KB
constexpr int kKeyChunk = 128;                         // keys per attention chunk: the rows of a tensor-core instruction
constexpr int kAttnBytesPerDim = 640;                  // attention tiles: 64 query rows, a chunk of keys and of values; bytes per column of a head
constexpr int kActSmemMax = 32768;                     // operand of a block's share of the down projection at most: its SwiGLU output, in pairs that of both blocks
constexpr int kPairSums = 65536;                       // partial sums per row from which on pairs of blocks share the down projection
constexpr int kMiscSmemBytes = 4096;
constexpr int kMiscOff = kSmemBudget - kMiscSmemBytes;  // bookkeeping lies behind everything else, at the same place whatever the rows
constexpr unsigned long long kLookaheadBytes = 393216;  // how far ahead of the ring the weight streamer reads into L2,
constexpr unsigned kLookaheadPiece = 8192;             //   in pieces of this size
constexpr int kLookaheadCycles = 600, kLookaheadSlow = 800;   //   and no more often than this: the slow rate
constexpr int kLookaheadRows = 24;                     //   above so many rows,
constexpr unsigned long long kLookaheadShare = 19ull << 17;   //   or where a block's share of a layer has more bytes (2.375 MB)
constexpr int kMaxDraftWords = 32;
constexpr int kProfWords = 12;                         // timestamps per (phase, block)
constexpr int kTmemCols = 512;
constexpr uint32_t kAccBufs = 4;                       // accumulator buffers: each two 128-row accumulators of up to 32 fp32 columns,
constexpr uint32_t kTmemBuf = 64;                      //   columns 0..255; so many that the issuing thread does not wait for a pass to be read out
constexpr uint32_t kTmemStack = 256;                   // stacked K slices (one pass, up to 256 columns): columns 256..511

enum OpIndex { OP_QKV = 0, OP_O = 1, OP_GU = 2, OP_DOWN = 3, OP_LM = 4, OP_RAW = 5, OP_COUNT = 6 };

struct OpDesc {
    int T;       // row tiles (16 weight rows each)
    int K16;     // column steps (16 input features each)
    int P_row;   // partitions along rows
    int P_k;     // partitions along columns (> 1: partial sums meet by reductions in L2)
    int rot;     // block index that owns partition 0 (spreads idle blocks over operations)
    int RW;      // row tiles per pass at most (16, 8, 4, 2 or 1)
    int SK;      // column steps per stage at most (RW * SK <= 64)
    int unit;    // row partitions are multiples of this many tiles (2 for gate|up: 16 SwiGLU columns)
    int follow;  // 1: the columns follow `gate|up`: one row partition, block i takes the columns that its partition i produces; or two (P_row
                 //   = 2), blocks 2 i and 2 i + 1 take half of the rows each and the columns that both of them produce
    int slices;  // K slices stacked as rows (0 or 1: none); divides K16 and the column shares
    unsigned long long w_off;  // byte offset of the operation inside its weight region
};

struct Part {
    int tile0, ntiles, k0, nk, pr, pk;
    unsigned long long off;  // byte offset of this partition from the operation's base
    int npass, nst;          // passes over the row tiles; stages per pass
    int pbase, prem;         // tiles per pass: pbase + (p < prem)
    int SK, slices;
    int per, rot;        // column steps per slice; pass the block begins with (it goes round from there)
};
// The i-th pass in the block's order.  Blocks whose partial sums meet in the same rows begin with different ones: reductions of all
// SMs into the same lines at the same moment take a quarter longer (55 KB of sums, all blocks: 4.9 us, begun apart 3.7).
__host__ __device__ inline int pass_index(const Part& p, int i) { return i + p.rot < p.npass ? i + p.rot : i + p.rot - p.npass; }
__host__ __device__ inline int pass_count(const Part& p, int i) { return p.pbase + (i < p.prem ? 1 : 0); }
__host__ __device__ inline int pass_start(const Part& p, int i) { return i * p.pbase + (i < p.prem ? i : p.prem); }

__host__ __device__ inline int even_start(int total, int parts, int i) {
    const int b = total / parts, r = total % parts;
    return i * b + (i < r ? i : r);
}
__host__ __device__ inline int even_count(int total, int parts, int i) {
    return total / parts + (i < total % parts ? 1 : 0);
}
// Inverse of even_start: which part holds element x.
__host__ __device__ inline int even_find(int total, int parts, int x) {
    const int b = total / parts, r = total % parts;
    if (x < r * (b + 1)) return x / (b + 1);
    return r + (x - r * (b + 1)) / b;
}

__host__ __device__ inline void finish_part(Part& p, const OpDesc& o) {
    p.off = (unsigned long long)kStepBytes *
            ((unsigned long long)p.tile0 * o.K16 + (unsigned long long)p.ntiles * p.k0);
    p.SK = o.SK;
    p.slices = o.slices > 1 ? o.slices : 1;
    p.npass = (p.ntiles + o.RW - 1) / o.RW;
    p.per = p.nk / p.slices;
    p.rot = 0;
    p.nst = (p.per + o.SK - 1) / o.SK;
    p.pbase = p.npass ? p.ntiles / p.npass : 0;
    p.prem = p.npass ? p.ntiles % p.npass : 0;
}

// Partition (pr, pk) of an operation; `gu` is the gate|up operation (used when o.follow).
__host__ __device__ inline Part make_part(const OpDesc& o, const OpDesc& gu, int pr, int pk) {
    Part p;
    p.pr = pr;
    p.pk = pk;
    if (o.follow) {
        const int units = gu.T / gu.unit;
        p.tile0 = even_start(o.T, o.P_row, pr);
        p.ntiles = even_count(o.T, o.P_row, pr);
        p.k0 = even_start(units, gu.P_row, pk * o.P_row);
        p.nk = even_start(units, gu.P_row, (pk + 1) * o.P_row) - p.k0;
    } else {
        p.tile0 = o.unit * even_start(o.T / o.unit, o.P_row, pr);
        p.ntiles = o.unit * even_count(o.T / o.unit, o.P_row, pr);
        p.k0 = even_start(o.K16, o.P_k, pk);
        p.nk = even_count(o.K16, o.P_k, pk);
    }
    finish_part(p, o);
    if (p.npass > 1 && (o.follow || o.P_k > 1)) p.rot = p.pk % p.npass;
    return p;
}

__host__ __device__ inline Part get_part(const OpDesc& o, const OpDesc& gu, int cta, int G) {
    const int rot = o.follow ? gu.rot : o.rot;
    const int nparts = o.follow ? gu.P_row : o.P_row * o.P_k;
    int idx = cta - rot;
    if (idx < 0) idx += G;
    if (idx >= nparts) {
        Part p;
        p.tile0 = p.ntiles = p.k0 = p.nk = p.pr = p.pk = p.npass = p.nst = p.pbase = p.prem = 0;
        p.SK = o.SK;
        p.slices = 1;
        p.per = p.rot = 0;
        p.off = 0;
        return p;
    }
    if (o.follow) return make_part(o, gu, idx % o.P_row, idx / o.P_row);
    return make_part(o, gu, idx / o.P_k, idx % o.P_k);
}

// Byte offset (from the operation's base) of the 16-byte unit holding columns 8*k8 .. 8*k8+7 of
// weight row `row`: the inverse view used when packing.
__host__ __device__ inline unsigned long long weight_offset(const OpDesc& o, const OpDesc& gu, int row, int k8) {
    const int t = row >> 4, ks = k8 >> 1, half = k8 & 1;
    int pr, pk;
    if (o.follow) {
        pr = even_find(o.T, o.P_row, t);
        pk = even_find(gu.T / gu.unit, gu.P_row, ks) / o.P_row;
    } else {
        pr = even_find(o.T / o.unit, o.P_row, t / o.unit);
        pk = even_find(o.K16, o.P_k, ks);
    }
    const Part p = make_part(o, gu, pr, pk);
    const int lt = t - p.tile0;
    const int pass = even_find(p.ntiles, p.npass, lt);
    const int start = pass_start(p, pass), pcount = pass_count(p, pass);
    const int tip = lt - start, lk = ks - p.k0;
    const int per = p.nk / p.slices, slice = lk / per, vk = lk % per;   // column steps per slice
    const int st = vk / p.SK, kin = vk % p.SK, v = pcount * p.slices;   // v: row tiles of the stage, slices stacked
    const unsigned long long stage_base =
        p.off + (unsigned long long)kStepBytes * ((unsigned long long)start * p.nk + (unsigned long long)v * st * p.SK);
    const unsigned long long in_stage =
        ((unsigned long long)(kin * 2 + half) * (2 * v) + ((slice * pcount + tip) * 2 + ((row & 15) >> 3))) * 128 + (row & 7) * 16;
    return stage_base + in_stage;
}

// What a block of a pair that may have abandoned a wait still has to see arrive before it leaves.  `mine`, `sent`: gate|up phases in which
// this block and the other one have sent their SwiGLU columns.  A phase is prepared for (bytes expected, all warps arrive) exactly where its columns
// are sent, and entered only once the phase before is over in the same block, so the two differ by one at most:
//   sent = mine - 1: the other block never sent the last phase's; those before have been waited for.
//   sent = mine:     the last phase's may be on their way (PAIR_LAST).
//   sent = mine + 1: the same, and those of a phase this block never prepared for (PAIR_NEXT).
enum PairDebt { PAIR_NONE = 0, PAIR_LAST = 1, PAIR_NEXT = 2 };
__host__ __device__ inline int pair_debt(int mine, int sent) {
    return (mine > 0 && sent >= mine ? PAIR_LAST : PAIR_NONE) | (sent > mine ? PAIR_NEXT : PAIR_NONE);
}

// Device state block (int32 words).
enum StateWord {
    ST_KV_LEN = 0, ST_HIST_LEN, ST_N_CTX, ST_PENDING, ST_DRAFT_LEN, ST_ACCEPT_LEN, ST_N_EMITTED, ST_ERR,
    ST_VERIFIED,      // 1 when a verify result awaits commit
    ST_MATCH_POS, ST_MATCH_LEN,
    ST_SEG_LEN,       // retained segment of rejected drafts (draft extension): tokens,
    ST_SEG_LIFE,      //   verify steps it has been appended to,
    ST_SEG_USED,      //   1 while it is part of the draft under verification,
    ST_BASE_LEN,      //   and that draft's length before it was appended
    ST_DB_LEN,        // tokens in the extra token database the drafter also searches (0: none)
    ST_DRAFT = 16,    // [32]
    ST_Y = 48,        // [33]
    ST_TREE_ON = 82,  // 1: the draft is a tree (ST_PARENT .. ST_ANC hold its shape), 0: a chain
    ST_PATH_LEN = 83, // nodes on the accepted path of the last tree verify
    ST_BUDGET = 84,   // tokens a run of enqueued steps may still emit (-1: no limit; 0: the remaining steps do nothing)
    ST_EMITTED = 96,  // [33]
    ST_SEG = 160,     // [32]
    ST_PARENT = 192,  // [32] row that row j continues (row 0 = the committed token; draft node i is row i)
    ST_DEPTH = 224,   // [32] distance of row j from the root = its position minus the KV length
    ST_ANC = 256,     // [32] bit r set: row r lies on row j's path from the root (j itself included)
    ST_PATH = 288,    // [32] accepted path (rows), root excluded
    ST_WORDS = 320
};

// Caller-supplied tokens (or other small whole numbers) by value, so that no host buffer has to outlive the call; n < 0: none.
struct DraftArg {
    int n;
    int tok[kMaxDraftWords];
};

// One sequence of a batched verify step: its rows [r0, r0 + M) of the launch, its committed length
// and its own KV cache.
struct BatchSeq {
    __nv_bfloat16* kcache;
    __nv_bfloat16* vcache;
    int r0, M, L, pad;
};

struct FwdParams {
    // model
    int n_layers, d, n_q, n_kv, hd, f, V, max_seq, g, n_qkv;
    float eps, scale_log2e;  // softmax scale 1/sqrt(hd) times log2(e)
    int G;                   // thread blocks in the grid
    OpDesc op[OP_COUNT];
    unsigned long long layer_stride;  // bytes of streamed weights per layer
    const uint8_t* wlayers;           // streamed weights of layer 0 (qkv, o, gate|up, down)
    const uint8_t* wlm;               // streamed LM head
    const uint8_t* wraw;              // streamed matrix of the stand-alone GEMM entry point
    const __nv_bfloat16* emb;         // [V][d] row-major (embedding gather)
    const float* norm_w;              // [n_layers][2][d], then the final norm [d]
    const float* bias;                // [n_layers][n_qkv] or nullptr
    const float2* rope;               // [max_seq][hd/2] (cos, sin)
    __nv_bfloat16* kcache;            // [layer][kv head][max_seq][hd]
    __nv_bfloat16* vcache;
    // activations (global, L2 resident)
    float* h;          // [kMaxRows][d] residual stream
    __nv_bfloat16* q;  // [kMaxRows][n_q * hd] queries, rotated
    float* part_o;     // [n_q][kMaxSplits][kMaxRows][hd] un-normalised split outputs
    float* part_ml;    // [n_q][kMaxSplits][kMaxRows][2]  (running max in log2 units, sum)
    float* cand_val;   // [G][kMaxRows] per-block best logit
    int* cand_idx;     // [G][kMaxRows] and its token id
    float* logits;     // [kMaxRows][V]
    const float* raw_x;  // [M][raw_K] operand of the stand-alone GEMM
    float* raw_out;    // [kMaxRows][raw_N] output of the stand-alone GEMM
    int raw_N, raw_K;
    int* state;
    const int* hist;
    unsigned* bar;     // grid barrier counter (wraps round; only differences are compared)
    unsigned long long* prof;  // optional [phase][block][kProfWords] timestamps (ns)
    // per launch
    int L;             // committed KV length = position of row 0
    int M;             // rows computed (1..kMaxRows)
    int NB;            // N of the tensor-core instruction: 16, or 32 when M > 16
    int att_gh;        // attention split: query heads per unit (the key ranges follow from it)
    int att_S, att_kps;  // key ranges and keys per range: derived from L and att_gh by the kernel when it starts
    int att_QG, att_per_seq;            // head groups per KV head; attention units per sequence
    int att_b0, att_hk0, att_qg0, att_s0;  // the block's first attention unit, decoded (each block works this out for itself)
    int mode;          // 0: rows are [pending, draft...]; 1: rows are hist[L..L+M)
    int ph_begin, ph_end;
    unsigned bar_base; // barrier counter value before this launch
    int store_logits;
    int tree;          // 1: the rows form a tree (positions, masks from the state block), 0: a chain
    // shared-memory plan of this launch (bytes from the 1024-aligned base)
    int nstage;        // ring slots of kStageBytes, at offset 0
    int u_off;         // operand region (token operand of the running GEMM; attention tiles)
    int act_off;       // SwiGLU output operand
    int p_off;         // exchange area of the q|k|v epilogue, probabilities of an attention unit
    int pad;           // 1: the rows of a column group in a token operand are followed by an empty one where that makes their number odd
    int plan_ks;       // what the plan follows from besides the rows: column steps of the widest token operand,
    int plan_act;      //   column steps of the down projection's operand at most (0: none)
    int plan_attn;     //   bytes the attention tiles need (0: no attention)
    int rows_from_state;  // 1: at most M rows; the draft in the state block says how many
    uint8_t att_gh_rows[kMaxRows];  // att_gh for 1, 2, ... rows (rows_from_state)
    unsigned long long wait_limit_ns;
    int l_from_state;  // 1: L is read from the state block when the kernel starts (steps enqueued without the host in between)
    // batched verify: nseq > 0 sequences share the launch (chains only); L is then the longest length
    int nseq;
    BatchSeq seq[kMaxBatch];
};

// Rows a column group of a token operand takes (`rows` token rows, K slices stacked).  An odd number spreads the groups over the
// banks: with a multiple of 8 every 16-byte unit of a token row lies in the same four banks, and the build's stores (one row,
// consecutive columns) take 16 turns instead of 2 (32 rows of 1536 columns: 8.6 -> 8.0 us a build).
__host__ __device__ inline int operand_rows(const FwdParams& P, int rows, int slices) {
    const int n = rows * (slices > 1 ? slices : 1);
    return P.pad ? n | 1 : n;
}
// Shared-memory plan of a launch over `rows` token rows: ring of weight stages | operand region | SwiGLU operand | bookkeeping (at
// kMiscOff).  The operand region holds the token operand of the widest GEMM share (or the attention
// tiles); the ring takes what is left.  Fewer than two ring slots: the rows do not fit.  The exchange area of the q|k|v
// epilogue and the probabilities of the attention step lie behind the attention tiles where the operand region is wide enough
// (the q|k|v operand there has been read by then if its blocks need one pass), else in the SwiGLU operand's place.
__host__ __device__ inline void plan_smem_rows(FwdParams& P, int rows) {
    for (P.pad = 1; P.pad >= 0; --P.pad) {
        const OpDesc& qkv = P.op[OP_QKV];
        const int step_bytes = 32 * operand_rows(P, rows, 1);  // token operand bytes per column step: 16 columns x rows x bf16
        int u = P.plan_ks * step_bytes;
        int act = P.plan_act * step_bytes;
        bool in_u = false;
        if (P.plan_attn > 0) {
            if (qkv.slices > 1) {
                const int q = qkv.K16 / qkv.slices * 32 * operand_rows(P, rows, qkv.slices);
                if (u < q) u = q;
            }
            if (u < P.plan_attn) u = P.plan_attn;
            int pr = (P.att_gh * rows + 15) & ~15;
            if (pr > 64) pr = 64;   // batched: a unit holds the rows of one sequence
            int scratch = 128 * (rows | 1) * 4;
            if (scratch < pr * kKeyChunk * 2) scratch = pr * kKeyChunk * 2;
            in_u = u >= P.plan_attn + scratch && (qkv.T + qkv.P_row - 1) / qkv.P_row <= qkv.RW;
            if (!in_u && act < scratch) act = scratch;
        }
        u = (u + 1023) / 1024 * 1024;
        act = act > 0 ? (act + 1023) / 1024 * 1024 : 1024;
        const int ring = kMiscOff - act - u;
        P.nstage = ring < 0 ? 0 : ring / kStageBytes;
        if (P.nstage > kMaxStages) P.nstage = kMaxStages;
        P.u_off = P.nstage * kStageBytes;
        P.act_off = P.u_off + u;
        P.p_off = in_u ? P.u_off + P.plan_attn : P.act_off;
        if (P.nstage >= 2 || P.pad == 0) return;
    }
}

}  // namespace sdv
