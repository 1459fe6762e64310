// The persistent MoE-layer megakernel: one CTA per SM, one launch per layer.
//
//   phase R  (all CTAs)   top-k routing of blocks of 4 to 64 tokens (32 to 4 threads per token),
//                         per-block expert bitmasks -> in-block ranks and a [block][expert]
//                         histogram; grid barrier (bounded; none up to 64 tokens)
//   set-up   (every CTA, redundantly) counts, offsets, candidate tile counts, cost model -> plan
//                         (c, K, n_steal), segment tables of the chosen K; permutation fix-up
//   phase A  (movement CTAs: blockIdx < c; every CTA in the phased plan)  x rows into expert-major Xe
//   phase B  (GEMM CTA pairs until the queue is empty; movement pairs for n_steal tiles)
//                         two neighbouring CTAs (a cluster of 2) share a tile of up to 256 rows: a scheduler
//                         warp claims tiles and waits for their inputs, TMA producers feed a
//                         6-stage smem ring, one thread issues tcgen05.mma.cta_group::2 into TMEM,
//                         four epilogue warps per CTA drain it through a staged, coalesced store,
//                         and a releasing warp makes the tiles' arrivals on the ready counters
//   phase C  (every CTA once it has nothing else)  combine tiles, chunk by chunk as the chunk's
//                         gemm1 tiles complete
//
// Stage list, roles, queue order, steal placement and the all-SM final combine follow the paper's
// Sections 3 and 4; the cost model is Section 3's Eq. 1-16.
#pragma once
#include <cuda.h>

#include <type_traits>

#include "weave_ptx.cuh"

namespace weave {

constexpr int kThreads = 256;
constexpr int kBM = 128;        // rows per GEMM m-block (UMMA M)
constexpr int kBK = 64;         // K elements per pipeline stage: 128 bytes of bf16 = one swizzle row
constexpr int kTN0 = 128;       // h columns per gemm0 tile; the MMA is N = 256 (gate | up)
constexpr int kStages = 6;
constexpr int kStageA = kBM * kBK * 2;                  // 16 KB: this CTA's 128 rows of A
constexpr int kStageB = 128 * kBK * 2;                  // 16 KB: this CTA's half (128 rows) of the 256-row B tile
constexpr int kStageBytes = kStageA + kStageB;          // 32 KB
constexpr int kEpiStageBytes = 4 * 4096;                // epilogue staging, per warp: 32 rows x 64 bytes (regular tiles); two 2 KB exchange buffers (swapped ones)
constexpr int kRouteBlock = 64;  // tokens per routing block (one 64-bit mask per expert)
constexpr int kLocalBlocks = 1;  // a batch of at most this many routing blocks is routed by every CTA for itself
                                 // (measured at two blocks: routing both in every CTA costs more than the grid barrier saves)
constexpr int kDirectTokens = 32; // largest batch whose gate/up tiles read x itself
constexpr int kCombTile = 16;    // tokens per combine tile (fewer when the batch would give fewer tiles than SMs)
constexpr int kMaxEE = 256;      // routed + shared experts
constexpr int kMaxTopK = 16;
constexpr int kFine = 8;         // fine chunks = largest chunk count K
constexpr int kMaxSeg = 1024;     // (chunk, expert) segments: K * (E+S) <= 1024 bounds the chunk count
constexpr int kTinfo = 2;        // tile-descriptor ring between the scheduler and its consumers.  Every slot is a tile claimed ahead;
                                 // pairs whose tiles share a weight panel stay closer together, and the last tiles are spread more
                                 // evenly, with two than with four (T = 8192 Qwen3-30B-shaped skewed 778 -> 757 us, Mixtral-shaped
                                 // 2457 -> 2421, T = 64 unchanged)
constexpr int kTmemCols = 512;
constexpr int kEpiWarps = 4;     // warps 4..7
constexpr int kRel = 3;          // mailbox ring between the epilogue warps and the releasing warp (warp 3)
constexpr unsigned kRelEnd = 0xFFFFFFFFu;
constexpr int kPairGroup = 8;    // row tiles of an expert kept L2-resident while all n-tiles pass

constexpr int kErrNonFinite = -5;
constexpr int kErrTimeout = -6;

enum { kModeAuto = 0, kModeFixed = 1, kModeSerial = 2 };

// Control words in global memory.  There are two sets of the words that a launch counts with (queues, flags, rows per
// chunk and expert), used in turn: a launch finds its own set zero and zeroes the other one, which the launch before it
// used, on its way in, so that nothing has to be cleaned up, and nobody has to be waited for, on the way out.  Which
// one is whose follows from `epoch`: CTA 0 adds 65536 - (CTAs - 1) as it leaves and every other CTA 1, so the upper half
// counts completed launches whatever their grids, and stays put until the last CTA of a launch is done.
// (Before, the last CTA out zeroed the words behind an atomic that every CTA waited for, and the static entry point
// zeroed its own with a memset: T = 1 40.1 -> 38.9 us, T = 64 200.7 -> 196.0, 8-expert T = 256 static 44.9 -> 41.3.)
struct CtlSet {
    unsigned bar_count;   // grid-barrier arrivals
    unsigned q_disp;      // next dispatch tile
    unsigned q_gemm[2];   // next GEMM tile (chunk-pipeline DAG order) of either list
    unsigned q_comb;      // next combine tile
    unsigned fix_done;    // routing blocks whose rows are final
    unsigned abort;       // set by the first wait that gives up; every wait polls it
    unsigned y_done[kFine];  // per chunk: epilogue-warp arrivals of finished gemm1 tiles
    unsigned q_pull;      // expert-parallel share: next block of remote tokens to stage
    unsigned pull_done;   // ... blocks staged
    unsigned x_local, x_in, x_in_uniq;   // ... the workload descriptors of Section 3.1, counted while routing
    unsigned pad[12];
    // followed by fcnt [8][256]: rows per (fine chunk, expert);
    //             xe_ready [nmb_max]: the row tile's rows that are dispatched;
    //             h_ready [nmb_max]: epilogue-warp arrivals of the row tile's gemm0 tiles
};
static_assert(sizeof(CtlSet) == 128, "the arrays behind it start on a line of their own");
__host__ __device__ __forceinline__ size_t ctl_set_bytes(int nmb_max)
{
    return (sizeof(CtlSet) + sizeof(unsigned) * ((size_t)kFine * kMaxEE + 2 * (size_t)nmb_max) + 255) / 256 * 256;
}
struct Ctl {
    unsigned epoch;
    unsigned pad[31];
    // results for the host
    int status;
    int timeout_where;
    int plan_c, plan_K, plan_steal;
    float plan_t;
    int plan_nmb, plan_ngemm;
    unsigned ep_x_local, ep_x_in, ep_x_in_uniq;
    int plan_kind;
};

// Plan kinds of the cost model.  kPlanSplit is the paper's (Eq. 15): c movement SMs beside N - c GEMM
// SMs from the start.  The other two exist because on one GPU the movement is an HBM copy that all
// SMs can do at full speed: kPlanDispatchAll lets every SM dispatch before the roles split (only the
// combine is left to the movement SMs), kPlanPhased has no roles at all (every SM dispatches, then
// runs GEMM tiles until the queue is empty, then combines; the ready flags still order the tiles,
// no grid barrier separates the phases).  kPlanRejoin is the split in which the movement SMs come back to
// the GEMM queue for good once the dispatch is done (no steal quota: they take GEMM tiles whenever no
// combine chunk is ready) and every GEMM CTA dispatches one m-block before its first tile; K = 1.
enum { kPlanSplit = 0, kPlanDispatchAll = 1, kPlanPhased = 2, kPlanRejoin = 3 };

struct KParams {
    int T, H, I, E, S, k, EE;
    int nblk;             // 64-token blocks = ceil(T / 64): the unit of the chunks, of small batches and of the expert-parallel share
    int lg_rb, nrb;       // routing blocks of 1 << lg_rb tokens, 4 to 64: as small as one block per CTA allows
    int mode, fixed_c, fixed_K, fixed_steal;
    int nt0, nt1;         // n-tiles per row tile: I / 128, ceil(H / 256)
    int nmb_max;          // allocated length of the flag arrays (row tiles are never more than m-blocks)
    int ep_rank, ep_size; // expert-parallel share (ep_size <= 1: off): this rank hosts experts
                          // [ep_rank*E/ep_size, (ep_rank+1)*E/ep_size) and owns token shard ep_rank
    int ep_tshard;        // tokens per shard = ceil(T / ep_size)
    __nv_bfloat16 *xs;    // [T][H] staging of remote tokens (each unique one is copied once)
    unsigned long long *uniq_mask;   // [nblk] remote tokens of the block that have a local expert
    int elastic_steal;    // movement pairs keep stealing past their quota while no combine chunk is ready
    int kinds;            // bit mask of the plan kinds the cost model may choose (bit kPlanSplit, ...)
    int direct;           // the gate/up tiles may read x itself (T <= kDirectTokens, see the kernel body); tm.x is set
    int withhold_mb;      // test hook: the rows of this m-block are never counted in (-1 = off)
    int c_min, c_max, c_step;
    float alpha;
    float eff[4];
    unsigned long long timeout_ns;
    const __nv_bfloat16 *x;
    const float *logits;
    __nv_bfloat16 *out;
    Ctl *ctl;
    uint8_t *sets;        // two CtlSets with their arrays, ctl_set_bytes(nmb_max) each
    int *hist;            // [nrb][256]; shares its place with xs, which only an expert-parallel share uses: every CTA waits
                          // for fix_done == nrb, and with it for the last look at hist, before it stages a row there
    int *topk_idx;        // [T][k]
    float *gates;         // [T][k]
    int *row_of;          // [T][k]
    int *token_of;        // [P]
    int *counts;          // [EE]
    int *offsets;         // [EE+1]
    __nv_bfloat16 *xe;    // [P][H]
    __nv_bfloat16 *hbuf;  // [P][I]
    __nv_bfloat16 *y;     // [P][H]
    const float *bw;      // [n_sm+1] byte/us
    const float *tf;      // [n_sm+1] FLOP/us
    uint4 *trace;         // optional [n_sm][trace_cap] event records (nullptr = off)
    int trace_cap;
    unsigned die_mask[32]; // bit smid: which half of the chip (die) the SM sits on
    int lists_pt;          // one chunk: two lists of GEMM tiles from this many row tiles on (see tile_lists_from)
    int4 *wait_log;       // [kWaitLogCtas][kWaitLogWarps]: written only by a wait that gives up or is cut short by the abort word
    float st_plan_t;      // weave_stream_kernel: the modelled time of its plan
};

struct TileInfo {
    int type;   // 0 gemm0 (+SwiGLU), 1 gemm1 of 256 rows, 2 no more tiles; 3 / 4 = gemm0 / gemm1 of a row tile of fewer
                // rows, with the operands swapped (weights on the MMA's M axis, the tile's rows on N)
    int mb;     // the m-block that this CTA's records name (row tile i of a segment stands for its m-blocks 2i, 2i + 1)
    int rt;     // row tile: the index of its ready flags
    int row0;   // first row of this CTA's 128 rows (regular) or of the tile (swapped)
    int nrows;  // valid rows from there
    int e, n, chunk, nkb;      // chunk | kTileLate: handed over before the tile's rows are there
};
constexpr int kTileLate = 256;

// what one movement buffer (a 32 KB stage) currently holds
struct MvDesc {
    int a;      // dispatch: first destination row        combine: token
    int b;      // dispatch: rows in the buffer            combine: first column
    int c;      // dispatch: m-block                       combine: columns
    int d;      // dispatch: 1 = last buffer of its tile;  2 = no more work (both phases);
                // 3 / 4 = staging of remote tokens (rows go to xs[tok[i]]; 4 = last buffer of the block)
    int n;      // combine: rows gathered (0: the token has no expert here, the piece is zero)
    float g[kMaxTopK + 8];   // combine: weight of each gathered row
    int tok[32];             // staging: destination token of each row in the buffer
};
constexpr int kMvBuf = kStageBytes;     // 32 KB
constexpr int kCombWarps = 6;           // warps 2..7 reduce

struct SmemTail {
    uint64_t full[kStages], empty[kStages];      // (the streaming kernel's rows of x and h reach over these 128 bytes)
    uint64_t tmem_full[2], tmem_empty[2];
    CtlSet *cs;                  // this launch's set of control words, and its arrays
    unsigned *fcnt, *xe_ready, *h_ready;
    uint64_t ti_full[kTinfo], ti_empty[kTinfo], ti_late[kTinfo];     // ti_late: the rows of a kTileLate tile are there
    uint64_t dv_full[kStages], dv_empty[kStages];   // dispatch: loader -> storer ring over the stage buffers
    uint64_t cb_full[kStages], cb_empty[kStages];   // combine: loader -> reducing warps
    uint64_t xg[2];                                 // swapped gemm0 epilogue: a gate and an up warp trade values
    uint64_t rel_full[kRel], rel_empty[kRel];       // epilogue warps -> releasing warp: a tile's stores are issued
    unsigned *rel_flag[kRel];                       // the ready counter that tile arrives on, and by how much
    unsigned rel_cnt[kRel];
    TileInfo ti[kTinfo];
    uint32_t tmem_base;
    int bcast[3];
    int red_i[8][4];
    float red_f[8];
    int scan_w[8];
    int scan_total;
    int c, K, steal, nmb, n_gemm, n_comb;
    int budget, die, direct;     // see gemm_phase
    int inline_disp;             // 1 = idle warps of the GEMM phase dispatch, 2 = and meet before their epilogues
    int elastic;                 // this launch: movement pairs take GEMM tiles beyond their quota, GEMM CTAs dispatch one m-block first
    int comb_tok;                // tokens per combine tile of this launch: 16, 8, 4, 2 or 1
    unsigned trace_n;
    int chunk_mb0[kFine + 1];
    int chunk_pt0[kFine + 1];
    int chunk_tile0[kFine + 1];
    int split_pt, split_seg;     // K = 1: pair tiles [0, split_pt) = segments [0, split_seg) are list 0, the rest list 1
    int offsets[kMaxEE + 1];
    int seg_mb0[kMaxSeg + 1];
    int seg_pt0[kMaxSeg + 1];    // prefix of row tiles: ceil(m-blocks / 2) per segment
    int seg_row0[kMaxSeg];
    int seg_rows[kMaxSeg];
};

// Scratch of the movement phases (dispatch, combine).  A CTA is in one phase at a time, so it shares
// its space with the second half of the GEMM epilogue's staging area.
struct MoveScratch {
    MvDesc mv[kStages];
    int tok[kBM];
    int crow[kCombTile][kMaxTopK + 8];
    float cgate[kCombTile][kMaxTopK + 8];
};
static_assert(sizeof(MoveScratch) <= kEpiStageBytes / 2, "movement scratch must fit half of the staging area");
// ... and of the dispatch in token order: destination row and row tile of every store out of a ring buffer
constexpr int kTokEnt = 128;
struct TokScratch {
    int n[kStages];                    // stores out of the buffer (-1: no more work)
    int row[kStages][kTokEnt], rt[kStages][kTokEnt];
};
static_assert(sizeof(TokScratch) <= kEpiStageBytes / 2, "as the movement scratch");
static_assert(kMaxTopK + 8 <= 32 && 32 <= kTokEnt, "a token's rows fit a buffer's list, and a warp");
static_assert(kLocalBlocks * (kMaxEE + 1) * 8 <= kEpiStageBytes / 2, "the routing masks must fit the other half");
static_assert(kLocalBlocks * kMaxEE * 8 <= 2048, "the masks end below the first upper exchange buffer, the only kind that tiles of at most 32 rows use");
static_assert(kDirectTokens <= 32, "gate/up tiles that read the masks stay out of the lower exchange buffers");
static_assert(kFine == 8, "chunk of a fine chunk = f >> (3 - log2 K)");
__device__ __forceinline__ MoveScratch &move_scratch(uint8_t *stages)
{
    return *reinterpret_cast<MoveScratch *>(stages + kStages * kStageBytes + kEpiStageBytes / 2);
}

constexpr int kSmemBytes = kStages * kStageBytes + kEpiStageBytes + (int)sizeof(SmemTail) + 1024;
static_assert(kSmemBytes <= 232448, "exceeds the 227 KB a CTA may opt into");

// [stage ring | epilogue staging | SmemTail], the ring on a 1024-byte boundary
__device__ __forceinline__ uint8_t *smem_stages()
{
    extern __shared__ uint8_t smem_raw[];
    return smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
}
__device__ __forceinline__ SmemTail &smem_tail()
{
    return *reinterpret_cast<SmemTail *>(smem_stages() + kStages * kStageBytes + kEpiStageBytes);
}

// ------------------------------------------------------------------------------------ waits

__device__ __noinline__ void give_up(Ctl *ctl, int where)
{
    if (atomicCAS(&ctl->status, 0, kErrTimeout) == 0) ctl->timeout_where = where;
    atomicExch(&smem_tail().cs->abort, 1u);
}

// Post-mortem of a failed launch: every wait that ends without success (its own limit ran out, or it saw
// the abort word another wait had raised) leaves {wait id, what it waited on (shared-memory address of the
// barrier or low bits of the flag's address), the parity or target it waited for, 1 = timed out / 2 = cut
// short} in its warp's slot (the warp's first such wait only).  Together the slots show who was waiting
// for whom when the launch stopped.
constexpr int kWaitLogCtas = 512, kWaitLogWarps = 16;      // (the streaming kernel has 16 warps; no sm_100 device has as many SMs)
__device__ __noinline__ void note_failed_wait(int4 *log, int where, unsigned what, unsigned want, int how)
{
    // the first failed wait of a warp is the one that tells where it stood; what it runs into afterwards,
    // on its way out with the abort word set, is not recorded  (no log for grids of more than kWaitLogCtas)
    int4 *slot = log + blockIdx.x * kWaitLogWarps + ((threadIdx.x >> 5) & (kWaitLogWarps - 1));
    if (log && slot->w == 0) *slot = make_int4(where, (int)what, (int)want, how);
}

// Optional timeline: one 16-byte record {start ns, end ns, kind<<24 | id, extra} per event, per CTA.
enum { kEvRoute = 1, kEvSetup = 2, kEvFixup = 3, kEvDispatch = 4, kEvGemmLoad = 5, kEvGemmEpi = 6,
       kEvCombine = 7, kEvWaitChunk = 8, kEvBarrier = 9, kEvMma = 11, kEvStream = 12 };
__device__ __forceinline__ void trace_ev(const KParams &p, SmemTail &S, int kind, unsigned id,
                                         unsigned long long t0, unsigned long long t1, unsigned extra)
{
    if (p.trace == nullptr) return;
    const unsigned i = atomicAdd(&S.trace_n, 1u);
    if (i + 1u < (unsigned)p.trace_cap)
        p.trace[(size_t)blockIdx.x * p.trace_cap + i] =
            make_uint4((unsigned)t0, (unsigned)t1, ((unsigned)kind << 24) | (id & 0xFFFFFFu), extra);
}
__device__ __forceinline__ unsigned long long trace_now(const KParams &p)
{
    return p.trace ? globaltimer_ns() : 0ull;
}
// the same for the CTA-wide phases, whose records thread 0 writes: the other threads do not read the timer
__device__ __forceinline__ unsigned long long trace_now_t0(const KParams &p)
{
    return (p.trace && threadIdx.x == 0) ? globaltimer_ns() : 0ull;
}

// Every wait is bounded: it polls the global abort word and a wall-clock limit, and returns false
// instead of spinning forever.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, const KParams &p, int where)
{
    if (mbar_try_wait(bar, parity)) return true;
    // the clock is read only every 32 polls (the first reading starts the limit): a reading costs far
    // more than a poll, and most waits end within a few polls.  The abort word is looked at one round
    // late: its load (an L2 round trip on a line that every SM's queue claims hit) is issued here and its
    // value used 32 polls later, so the waiting thread is never stalled on it when the barrier completes.
    unsigned long long t0 = 0;
    unsigned it = 0;
    unsigned ab = 0u;
    while (!mbar_try_wait(bar, parity)) {
        if ((++it & 31u) == 0u) {
            if (ab) { note_failed_wait(p.wait_log, where, smem_u32(bar), parity, 2); return false; }
            ab = ld_relaxed_u32(&smem_tail().cs->abort);
            const unsigned long long now = globaltimer_ns();
            if (t0 == 0) t0 = now;
            else if ((long long)(now - t0) > (long long)p.timeout_ns) {     // signed: a timer that steps back is not a time-out
                give_up(p.ctl, where);
                note_failed_wait(p.wait_log, where, smem_u32(bar), parity, 1);
                return false;
            }
        }
    }
    return true;
}

__device__ __forceinline__ bool flag_wait_ge(const unsigned *flag, unsigned target, const KParams &p, int where)
{
    if (ld_acquire_u32(flag) >= target) return true;
    unsigned long long t0 = 0;
    unsigned it = 0;
    while (ld_acquire_u32(flag) < target) {
        __nanosleep(40);
        if ((++it & 31u) == 0u) {
            if (ld_relaxed_u32(&smem_tail().cs->abort)) {
                note_failed_wait(p.wait_log, where, (unsigned)(size_t)flag, target, 2);
                return false;
            }
            const unsigned long long now = globaltimer_ns();
            if (t0 == 0) t0 = now;
            else if ((long long)(now - t0) > (long long)p.timeout_ns) {
                give_up(p.ctl, where);
                note_failed_wait(p.wait_log, where, (unsigned)(size_t)flag, target, 1);
                return false;
            }
        }
    }
    return true;
}

__device__ __forceinline__ void linger_after_abort()
{
    // lets copies and MMAs that are already in flight land before this CTA can leave
    const unsigned long long t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 50000ull) __nanosleep(1000);
}

// All CTAs are co-resident (cooperative launch); arrivals accumulate over the barriers of a launch.
// Two exclusive scans in one pass: v = a | b << 32.
__device__ __forceinline__ unsigned long long block_excl_scan_packed(unsigned long long v, SmemTail &S, unsigned long long &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += n;
    }
    __syncthreads();
    if (lane == 31) { S.red_i[warp][0] = (int)(unsigned)inc; S.red_i[warp][1] = (int)(unsigned)(inc >> 32); }
    __syncthreads();
    unsigned long long wbase = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        const unsigned long long sw = (unsigned long long)(unsigned)S.red_i[w][0] | ((unsigned long long)(unsigned)S.red_i[w][1] << 32);
        if (w < warp) wbase += sw;
        tot += sw;
    }
    total = tot;
    return wbase + inc - v;
}

// the two halves of a grid barrier, for a caller that has work to do between arriving and waiting
__device__ __forceinline__ void grid_barrier_arrive(SmemTail &S)
{
    __syncthreads();      // (the release is cumulative: it covers what the other threads wrote before the block barrier)
    if (threadIdx.x == 0) red_release_add_u32(&S.cs->bar_count, 1u);
}
__device__ __forceinline__ bool grid_barrier_wait(const KParams &p, SmemTail &S, unsigned target, int where)
{
    if (threadIdx.x == 0) S.bcast[2] = flag_wait_ge(&S.cs->bar_count, target, p, where) ? 1 : 0;
    __syncthreads();
    return S.bcast[2] != 0;
}
__device__ __forceinline__ bool grid_barrier(const KParams &p, SmemTail &S, unsigned target, int where)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        red_release_add_u32(&S.cs->bar_count, 1u);
        S.bcast[2] = flag_wait_ge(&S.cs->bar_count, target, p, where) ? 1 : 0;
    }
    __syncthreads();
    return S.bcast[2] != 0;
}

// ------------------------------------------------------------------------------------ block helpers

__device__ __forceinline__ int block_excl_scan(int v, SmemTail &S, int &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += n;
    }
    __syncthreads();
    if (lane == 31) S.scan_w[warp] = inc;
    __syncthreads();
    int wbase = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
        int s = S.scan_w[w];
        if (w < warp) wbase += s;
        tot += s;
    }
    total = tot;
    return wbase + inc - v;
}

// ------------------------------------------------------------------------------------ phase R

// Four threads route one token, so a CTA's 256 threads take a whole 64-token block at once and every
// warp instruction serves eight tokens (a prologue of eight warps per SM is bound by the instructions each
// warp has to issue, not by their latencies).  The block's logits are staged in shared memory (row stride
// = 4 mod 32 words, so the 32 lanes of a warp - eight tokens x four threads - hit 32 different banks).
// Thread q of a quad holds experts q, q+4, ... as order keys in registers; the k selections are k rounds of
// arg-max over the quad.  Order: larger logit first, equal logits by lower expert index (-0 == +0);
// gates = softmax over the selected k.

// fp32 -> uint32 that orders like the float (finite values; -0 has been folded into +0)
__device__ __forceinline__ unsigned float_order_key(float v)
{
    const unsigned u = __float_as_uint(v);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float float_from_order_key(unsigned k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

__device__ __forceinline__ int route_row_stride(int E) { return ((E + 27) / 32) * 32 + 4; }

// cooperative copy of the block's logit rows into shared memory, coalesced; all copies are in flight
// together (one memory round trip).  The caller waits (cp_async_wait_all) and publishes them
// (__syncthreads) when it needs them, and may do other work in between.
__device__ __forceinline__ void stage_logits_issue(const KParams &p, int b, float *lg_s)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t0 = b << p.lg_rb, ntok = min(1 << p.lg_rb, p.T - t0);
    const int stride = route_row_stride(p.E);
    if ((p.E & 3) == 0) {      // rows are 16-byte multiples: both sides of every copy are 16-byte aligned
        const int per_row = p.E >> 2;
        for (int i = threadIdx.x; i < ntok * per_row; i += kThreads) {
            const int r = i / per_row, c = (i - r * per_row) << 2;
            cp_async_16(smem_u32(lg_s + r * stride + c), p.logits + (size_t)(t0 + r) * p.E + c);
        }
    } else {
        for (int r = warp; r < ntok; r += kThreads / 32) {
            const float *src = p.logits + (size_t)(t0 + r) * p.E;
            for (int c = lane; c < p.E; c += 32) cp_async_4(smem_u32(lg_s + r * stride + c), src + c);
        }
    }
}

// Top-k selection of routing block b by k rounds of arg-max.  Thread q of a quad owns experts q, q+4, ...
// of its token.  A first pass turns the staged logits into order keys IN PLACE (shared memory) and finds
// the thread's best (largest key, lowest expert index among equals).  A round: the quad's best of the four
// bests (two shuffle steps; equal keys go to the lower expert index) is slot j; its owner writes a zero over
// that key and rescans its keys.  The keys live in shared memory rather than in registers so that both
// passes are short ROLLED loops: this code runs once or twice per launch, at the speed of instruction
// fetch, and a loop body is fetched once (the unrolled register version issued fewer instructions and
// took twice as long).  The scratch arrays come as 32-bit shared-memory addresses.  r_mask[e] (64 bits):
// bit tl set when token tl of the block selected expert e (an expert hosted here); r_idx[tl][j]: the
// expert of slot j, -1 when another rank hosts it; r_cnt: local / remote (token, expert) pairs of the
// block (expert-parallel share only); r_p: [64][16] floats of scratch for the exponentials (the sum is
// only known once all k slots are chosen).  write_out: this CTA is the one that writes the block's selections
// and gates to global memory (every CTA routes a small batch for itself, one of them writes it down).
// Its shared-memory accesses name the shared space, so that it could also be compiled out of line (a function
// that is not inlined sees generic pointers, and generic atomics that land in shared memory take a slow
// path); inlined it is 1-3 us per layer faster on the small batches.
struct RouteArgs {
    int lg_rb, T, E, k, ep_size, ep_rank, ep_tshard;
    int *status;
    int *topk_idx;
    float *gates;
};
// kQuad: 64-token blocks, four threads per token.  Otherwise 32 to 4 tokens with 8, 16 or 32 threads each: a thread
// then goes through E / 8 to E / 32 experts instead of E / 4 (routing of a block, staging included: E = 256, k = 8, T = 1023 12.5 -> 7.4 us, E = 128, T = 1 7.8 -> 5.8).
template <bool kQuad>
__device__ __forceinline__ void route_block(int lg_rb, int T, int E, int k, int ep_size, int ep_rank, int ep_tshard, int *status,
                                               int *topk_idx, float *gates, int b, uint32_t lg_s, uint32_t r_mask,
                                               uint32_t r_idx, uint32_t r_cnt, uint32_t r_p, bool write_out)
{
    static_assert(kThreads == 4 * kRouteBlock, "four threads per token of a 64-token routing block");
    const int lg = kQuad ? 2 : min(5, 8 - lg_rb), G = 1 << lg;      // G threads per token
    const int tl = threadIdx.x >> lg, q = threadIdx.x & (G - 1);
    const int t = (b << (kQuad ? 6 : lg_rb)) + tl;
    const bool valid = t < T && (kQuad || tl < (1 << lg_rb));
    const int e_lo = ep_size > 1 ? ep_rank * (E / ep_size) : 0;
    const int e_hi = ep_size > 1 ? e_lo + E / ep_size : E;
    const uint32_t row = lg_s + 4u * (uint32_t)(tl * route_row_stride(E));      // this token's logits, then keys

    if (!__any_sync(0xffffffffu, valid)) return;      // (a warp without a token)
    // keys: 0 = nothing there; every finite logit maps to a key >= 1 that orders like the float
    // (a token past the end keeps all-zero keys: its quad then selects nothing and writes nothing)
    unsigned bk = 0u;
    int be = 0x7fffffff;      // expert of this thread's best key
    bool bad = false;
#pragma unroll 2
    for (int e = q; e < E; e += G) {
        float x = ld_shared_f32(row + 4u * (uint32_t)e);
        const bool nf = !(fabsf(x) <= 3.402823466e38f);      // NaN or +-inf: flag it, keep indices in range
        bad = bad || (valid && nf);
        x = nf ? -3.402823466e38f : x;
        x = __fadd_rn(x, 0.0f);                              // folds -0 into +0, leaves everything else alone
        const unsigned c = valid ? float_order_key(x) : 0u;
        st_shared_u32(row + 4u * (uint32_t)e, c);
        if (c > bk) { bk = c; be = e; }                      // strict: the lower expert index stays
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicCAS(status, 0, kErrNonFinite);

    float vmax = 0.f, sum = 0.f;
    int nloc = 0;
    for (int j = 0; j < k; ++j) {
        unsigned hk = bk;
        int hi = bk ? be : 0x7fffffff;
        if (!kQuad && lg == 5) {      // a whole warp per token: two reductions in hardware
            const unsigned top = __reduce_max_sync(0xffffffffu, hk);
            hi = (int)__reduce_min_sync(0xffffffffu, hk == top ? (unsigned)hi : 0x7fffffffu);
            hk = top;
        } else {
#pragma unroll kQuad ? 2 : 1
            for (int o = 1; o < G; o <<= 1) {
                const unsigned ok = __shfl_xor_sync(0xffffffffu, hk, o);
                const int oi = __shfl_xor_sync(0xffffffffu, hi, o);
                if (ok > hk || (ok == hk && oi < hi)) { hk = ok; hi = oi; }
            }
        }
        // every thread of the quad knows slot j now; thread j mod 4 writes it down
        const float v = float_from_order_key(hk);
        if (j == 0) vmax = v;
        const float pj = expf(v - vmax);
        sum += pj;                                   // slot order
        // expert-parallel share: only the experts hosted here get rows; the gates stay normalised over
        // all k selected experts
        const bool local = hi >= e_lo && hi < e_hi;
        nloc += local ? 1 : 0;
        if (valid && (j & (G - 1)) == q) {
            st_shared_u32(r_p + 4u * (uint32_t)(tl * kMaxTopK + j), __float_as_uint(pj));
            if (write_out) {
                topk_idx[(size_t)t * k + j] = hi;
                st_shared_u32(r_idx + 4u * (uint32_t)(tl * kMaxTopK + j), (uint32_t)(local ? hi : -1));
            }
            if (local) red_shared_or_u32(r_mask + 8u * (uint32_t)hi + 4u * (uint32_t)(tl >> 5), 1u << (tl & 31));
        }
        // the owner takes its winner out and looks for its next best
        if ((hi & (G - 1)) == q && hk != 0u) {
            st_shared_u32(row + 4u * (uint32_t)hi, 0u);
            bk = 0u; be = 0x7fffffff;
#pragma unroll 4
            for (int e = q; e < E; e += G) {
                const unsigned c = ld_shared_u32(row + 4u * (uint32_t)e);
                if (c > bk) { bk = c; be = e; }
            }
        }
    }
    __syncwarp();
    if (valid) {
        if (write_out)
            for (int j = q; j < k; j += G)
                gates[(size_t)t * k + j] = __fdiv_rn(__uint_as_float(ld_shared_u32(r_p + 4u * (uint32_t)(tl * kMaxTopK + j))), sum);
        if (ep_size > 1 && q == 0 && nloc) {
            if (t / ep_tshard == ep_rank) red_shared_add_u32(r_cnt, (uint32_t)nloc);
            else {
                red_shared_add_u32(r_cnt + 4u, (uint32_t)nloc);
                red_shared_or_u32(r_mask + 8u * (uint32_t)kMaxEE + 4u * (uint32_t)(tl >> 5), 1u << (tl & 31));
            }
        }
    }
}

// ------------------------------------------------------------------------------------ cost model

// Eq. 15 for one candidate, in the same fp32 operation order as the CPU restatement:
// T_comp = W_comp / (TFLOPS(N-c) * eff_chunk(K))  (Eq. 9),  T_comm = (W_disp + W_comb) / BW(c)  (Eq. 5),
// T_tail = (1 - alpha) * W_comb / (BW(c) * K)  (Eq. 10),  T_total = max(T_comp + T_tail, T_comm).
// bw = BW(c), tf = TFLOPS(N - c): the candidate's two table entries
template <class PB>
__device__ __forceinline__ float model_t_total(const PB &p, float bw, float tf, int ki, float w_comp, float w_disp,
                                               float w_comb)
{
    const float Kf = (float)(1 << ki);
    const float t_comp = __fdiv_rn(w_comp, __fmul_rn(tf, p.eff[ki]));
    const float t_comm = __fdiv_rn(__fadd_rn(w_disp, w_comb), bw);
    const float t_tail = __fmul_rn(__fsub_rn(1.0f, p.alpha), __fdiv_rn(w_comb, __fmul_rn(bw, Kf)));
    return fmaxf(__fadd_rn(t_comp, t_tail), t_comm);
}

// Plan kind "dispatch on all SMs, then split": W_disp / BW(N), then Eq. 15 with only the combine left as
// communication.  bw_n = BW(N).
template <class PB>
__device__ __forceinline__ float model_t_dispatch_all(const PB &p, float bw, float tf, float bw_n, int ki, float w_comp,
                                                      float w_disp, float w_comb)
{
    const float Kf = (float)(1 << ki);
    const float t_disp = __fdiv_rn(w_disp, bw_n);
    const float t_comp = __fdiv_rn(w_comp, __fmul_rn(tf, p.eff[ki]));
    const float t_tail = __fmul_rn(__fsub_rn(1.0f, p.alpha), __fdiv_rn(w_comb, __fmul_rn(bw, Kf)));
    const float t_comb = __fdiv_rn(w_comb, bw);
    return __fadd_rn(t_disp, fmaxf(__fadd_rn(t_comp, t_tail), t_comb));
}

// Plan kind "phased": dispatch, GEMMs and combine one after the other, each on all N SMs.
template <class PB>
__device__ __forceinline__ float model_t_phased(const PB &p, float bw_n, float tf_n, float w_comp, float w_disp, float w_comb)
{
    return __fadd_rn(__fadd_rn(__fdiv_rn(w_disp, bw_n), __fdiv_rn(w_comp, tf_n)),
                     __fmul_rn(__fsub_rn(1.0f, p.alpha), __fdiv_rn(w_comb, bw_n)));
}

// Plan kind "split with rejoin": while c SMs dispatch (W_disp / BW(c)), N - c SMs run GEMM tiles (the work
// done meanwhile as in Eq. 12, but no more than the gate/up tiles of the layer, 4HI of the 6HI FLOPs per
// row: the queue runs them first and a down tile needs its m-block's gate/up tiles, so a dispatch that
// outlasts them holds the GEMM SMs up); what is left then runs on all N SMs; the final combine is on all
// N SMs.
template <class PB>
__device__ __forceinline__ float model_t_rejoin(const PB &p, float bw, float tf, float bw_n, float tf_n, float w_comp,
                                                float w_disp, float w_comb)
{
    const float t_disp = __fdiv_rn(w_disp, bw);
    const float w_during = fminf(__fmul_rn(t_disp, tf), __fmul_rn(w_comp, 0.6666667f));
    const float w_rest = fmaxf(0.0f, __fsub_rn(w_comp, w_during));
    return __fadd_rn(__fadd_rn(t_disp, __fdiv_rn(w_rest, tf_n)),
                     __fmul_rn(__fsub_rn(1.0f, p.alpha), __fdiv_rn(w_comb, bw_n)));
}

// Eq. 11-14 with W_tile = W_comp / n_tiles (the mean GEMM tile of this layer).
__device__ __forceinline__ int model_n_steal(int n_sm, float bw, float tf, float w_comp, float w_disp,
                                             float w_comb, int n_tiles)
{
    if (n_tiles <= 0) return 0;
    const float t_comm = __fdiv_rn(__fadd_rn(w_disp, w_comb), bw);
    const float w_partial = __fmul_rn(t_comm, tf);
    const float w_steal = fmaxf(0.0f, __fsub_rn(w_comp, w_partial));
    const float w_tile = __fdiv_rn(w_comp, (float)n_tiles);
    if (!(w_tile > 0.0f)) return 0;
    // a GEMM worker is a CTA pair: W_steal is shared by n_sm / 2 workers (Eq. 14's N)
    const float ns = __fdiv_rn(w_steal, __fmul_rn((float)(n_sm / 2), w_tile));
    int r = (int)floorf(__fadd_rn(ns, 0.5f));
    return max(0, min(r, n_tiles));
}

// Eq. 16: the arg-min of the modelled layer time over the candidate plans, evaluated by the whole CTA (every
// CTA evaluates it for itself and gets the same answer).  Thread tid owns the split candidate
// (c, K) = (c_min + (tid >> 2) * c_step, 1 << (tid & 3)) and its "dispatch on all SMs first" and "rejoin"
// variants; thread 0 also owns the phased plan.  Candidate order = (kind, c ascending, K ascending),
// index = kind * 256 + thread; the phased plan is index 512, the rejoin plans follow it; ties go to the
// smaller index.  Contains one __syncthreads(); S.red_f and S.red_i[.][0] carry the reduction.
struct PlanPick { int c, ki, kind; float t; };
struct ModelArgs { float alpha, eff[4]; int kinds, c_min, c_step; };     // by value, see RouteArgs
__device__ __noinline__ PlanPick model_pick(const ModelArgs p, SmemTail &S, int n_sm, float w_comp, float w_disp, float w_comb,
                                            bool cm_ok, float cm_bw, float cm_tf, float cm_bw_n, float cm_tf_n)
{
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cm_ki = tid & 3;
    float t = __int_as_float(0x7f800000);
    int bi = tid;
    if (cm_ok && (p.kinds & (1 << kPlanSplit))) t = model_t_total(p, cm_bw, cm_tf, cm_ki, w_comp, w_disp, w_comb);
    if (cm_ok && (p.kinds & (1 << kPlanDispatchAll))) {
        const float t1 = model_t_dispatch_all(p, cm_bw, cm_tf, cm_bw_n, cm_ki, w_comp, w_disp, w_comb);
        if (t1 < t) { t = t1; bi = kThreads + tid; }
    }
    if (tid == 0 && (p.kinds & (1 << kPlanPhased))) {
        const float t2 = model_t_phased(p, cm_bw_n, cm_tf_n, w_comp, w_disp, w_comb);
        if (t2 < t) { t = t2; bi = 2 * kThreads; }
    }
    if (cm_ok && cm_ki == 0 && (p.kinds & (1 << kPlanRejoin))) {      // K = 1 only
        const float t3 = model_t_rejoin(p, cm_bw, cm_tf, cm_bw_n, cm_tf_n, w_comp, w_disp, w_comb);
        if (t3 < t) { t = t3; bi = 3 * kThreads + tid; }
    }
    // (rolled loops: this code runs once per launch, at the speed of instruction fetch)
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) {
        const float ot = __shfl_xor_sync(0xffffffffu, t, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ot < t || (ot == t && oi < bi)) { t = ot; bi = oi; }
    }
    if (lane == 0) { S.red_f[warp] = t; S.red_i[warp][0] = bi; }
    __syncthreads();
    t = S.red_f[0]; bi = S.red_i[0][0];
#pragma unroll 1
    for (int w = 1; w < kThreads / 32; ++w) {
        const float ot = S.red_f[w];
        const int oi = S.red_i[w][0];
        if (ot < t || (ot == t && oi < bi)) { t = ot; bi = oi; }
    }
    PlanPick r;
    r.kind = bi / kThreads;
    const int bt = bi % kThreads;      // the thread that evaluated the winner
    r.c = r.kind == kPlanPhased ? n_sm : p.c_min + (bt >> 2) * p.c_step;
    r.ki = r.kind == kPlanPhased ? 0 : (bt & 3);
    r.t = t;
    return r;
}

// ------------------------------------------------------------------------------------ tile decoding

// largest s in [lo, hi) with (seg_mb0[s] - base) * mul <= key   (empty segments share a start)
__device__ __forceinline__ int seg_search(const SmemTail &S, int lo, int hi, int base, int mul, int key)
{
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if ((S.seg_mb0[mid] - base) * mul <= key) lo = mid; else hi = mid;
    }
    return lo;
}

// m-block -> its rows; seg = the (chunk, expert) segment it belongs to (index chunk * EE + expert)
__device__ __forceinline__ void decode_mblock(const SmemTail &S, int EE, int mb, int &row0, int &nrows, int &seg)
{
    const int s = seg_search(S, 0, S.K * EE, 0, 1, mb);
    seg = s;
    const int m = mb - S.seg_mb0[s];
    row0 = S.seg_row0[s] + m * kBM;
    nrows = min(kBM, S.seg_rows[s] - m * kBM);
}

// A segment of R rows is worked on as ceil(R / 256) row tiles of almost equal size, in units of 16 rows (the MMA's N comes
// in sixteens): the first ones have a unit more.  A tile of 256 rows runs as a regular tile, rows on the MMA's M axis;
// any other runs swapped, weights on M and its 16 to 240 rows on N, so that it costs what its rows cost.  (With regular
// tiles of 256 rows and a swapped one for the rest, eight rows over a multiple of 256 cost two thirds of a tile for
// every panel of weights: Mixtral-shaped layer, T = 4096, 1014-1049 rows per expert 2117 us, 1024 each 1923.)
__host__ __device__ __forceinline__ void rowtile_span(int rows, int pts, int i, int &first, int &n)
{
    const int units = (rows + 15) >> 4, q = units / pts, r = units - q * pts;
    const int u0 = i * q + (i < r ? i : r), nu = q + (i < r ? 1 : 0);
    first = u0 << 4;
    n = nu << 4;
    if (first + n > rows) n = rows - first;
}
// the row tile that row `rel` of a segment belongs to
__host__ __device__ __forceinline__ int rowtile_of_rel(int rows, int pts, int rel)
{
    if (pts <= 1) return 0;
    const int units = (rows + 15) >> 4, q = units / pts, r = units - q * pts, u = rel >> 4;
    return u < r * (q + 1) ? u / (q + 1) : r + (u - r * (q + 1)) / q;
}

// GEMM queue order (the chunk-pipeline DAG order): chunk by chunk; inside a chunk all gemm0 tiles,
// then all gemm1 tiles (every gemm0 tile a gemm1 tile waits for comes earlier in the queue and waits
// only for dispatch, which keeps the in-order schedulers free of deadlock); inside those
// expert-major, then groups of kPairGroup pair tiles, n-tile, pair tile fastest: consecutive tiles
// share a weight panel, and a group's rows stay in L2 while all its n-tiles pass.  A pair tile = one row tile of a
// segment, for one n-tile.  `lead` describes the leader CTA's half, `peer` the other CTA's.
// Two other orders were measured and dropped: spreading the swapped tiles evenly over the queue
// (no faster, and a large expert's panels were fetched a second time for its last m-block: +27 %
// DRAM traffic on the Mixtral-shaped layer), and alternating gemm1 with gemm0 units (+1 % at
// I = 512, -9 % on the Qwen3-235B-shaped stack: two weight working sets in L2).
// Host-callable so that the order can be checked without a GPU.
// With one chunk the queue is cut into two lists at an expert's boundary (split_seg), one for each half of the
// chip, see the set-up; `list` says which one g counts in.
__host__ __device__ __forceinline__ void decode_pair_tile(const SmemTail &S, const KParams &p, int list, int g, TileInfo &lead,
                                                          TileInfo &peer)
{
    int j = 0, local = g, cpt0, nptj, lo, hi;
    if (S.K == 1) {
        cpt0 = list ? S.split_pt : 0;
        nptj = (list ? S.chunk_pt0[1] : S.split_pt) - cpt0;
        lo = list ? S.split_seg : 0;
        hi = list ? p.EE : S.split_seg;
    } else {
        while (j + 1 < S.K && g >= S.chunk_tile0[j + 1]) ++j;
        local = g - S.chunk_tile0[j];
        cpt0 = S.chunk_pt0[j];
        nptj = S.chunk_pt0[j + 1] - cpt0;
        lo = j * p.EE;
        hi = lo + p.EE;
    }
    int type = 0, nt = p.nt0;
    if (local >= nptj * p.nt0) { type = 1; local -= nptj * p.nt0; nt = p.nt1; }
    // largest s of the list with (seg_pt0[s] - cpt0) * nt <= local (empty segments share a start)
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if ((S.seg_pt0[mid] - cpt0) * nt <= local) lo = mid; else hi = mid;
    }
    const int s = lo;
    const int pts = S.seg_pt0[s + 1] - S.seg_pt0[s];
    const int within = local - (S.seg_pt0[s] - cpt0) * nt;
    const int gi = within / (kPairGroup * nt);
    const int wg = within - gi * kPairGroup * nt;
    const int gsize = (pts - gi * kPairGroup) < kPairGroup ? (pts - gi * kPairGroup) : kPairGroup;
    const int n = wg / gsize;
    const int ti = gi * kPairGroup + (wg - n * gsize);
    const int rows = S.seg_rows[s], mbs = S.seg_mb0[s + 1] - S.seg_mb0[s];
    int first, nr;
    rowtile_span(rows, pts, ti, first, nr);
    lead.type = type;
    lead.e = s - j * p.EE;
    lead.n = n;
    lead.chunk = j;
    lead.nkb = (type == 0 ? p.H : p.I) / kBK;
    lead.rt = S.seg_pt0[s] + ti;
    lead.mb = S.seg_mb0[s] + 2 * ti;
    lead.row0 = S.seg_row0[s] + first;
    lead.nrows = nr;
    const bool regular = nr > 240;      // 16 units, the last of them perhaps not full
    if (!regular) lead.type = type + 3;
    peer = lead;
    if (2 * ti + 1 < mbs) peer.mb = lead.mb + 1;
    if (regular) {
        lead.nrows = kBM;
        peer.row0 += kBM;
        peer.nrows -= kBM;
    }
}

// epilogue-warp arrivals on y_done[j] when all gemm1 tiles of chunk j are finished: both CTAs' warps for every tile
__device__ __forceinline__ unsigned y_done_target(const SmemTail &S, const KParams &p, int j)
{
    return (unsigned)((S.chunk_pt0[j + 1] - S.chunk_pt0[j]) * p.nt1 * 2 * kEpiWarps);
}

// ------------------------------------------------------------------------------------ phase A: dispatch

// Tile = one m-block: Xe[row0 + r] = x[token_of[row0 + r]].  The copy engine does the moving: warp 0
// gathers the source rows with bulk loads into a ring of 32 KB buffers, one thread of warp 1
// writes each full buffer to its (contiguous) destination rows with one bulk store.  About 96 KB
// of loads and as much of stores are in flight per SM.  The m-block's ready flag is released once
// its last store has completed.
// n_disp = number of CTAs that take part in the dispatch of this launch: CTA i's first tile is m-block i
// (no queue round trip before the first copy), later claims go through the queue, which starts at n_disp.
// local_route (a small batch that every CTA routed for itself): this CTA's copy of the routing blocks'
// expert masks, [nblk][kMaxEE + 1], sits at the start of the epilogue staging area; the source tokens of a
// tile are looked up there and nothing is read from the routing outputs in global memory.
__device__ __forceinline__ int nth_set_bit(unsigned long long m, int r)
{
    const unsigned lo = (unsigned)m, hi = (unsigned)(m >> 32);
    const int cl = __popc(lo);
    return r < cl ? (int)__fns(lo, 0u, r + 1) : 32 + (int)__fns(hi, 0u, r - cl + 1);
}
__device__ __forceinline__ void dispatch_phase(const KParams &p, SmemTail &S, uint8_t *stages, int max_tiles, int n_disp,
                                               bool local_route)
{
    const unsigned long long *lmask = local_route ? reinterpret_cast<const unsigned long long *>(stages + kStages * kStageBytes) : nullptr;
    MoveScratch &M = move_scratch(stages);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    fence_proxy_async_shared();      // the buffers held routing scratch written with ordinary stores
    __syncthreads();
    const uint32_t rowb = (uint32_t)p.H * 2u;
    const int R = max(1, kMvBuf / (int)rowb);     // rows per buffer
    if (warp == 0) {
        // ---- loader
        int b = 0;
        uint32_t ph = 0;
        bool ok = true;
        if (lane == 0 && lmask == nullptr) ok = flag_wait_ge(&S.cs->fix_done, (unsigned)p.nrb, p, 10);
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (p.ep_size > 1) {
            // expert-parallel share: first every remote token that has an expert here is copied ONCE
            // into the staging buffer xs (the dispatch-side deduplication of the paper's Section 4);
            // the rows of all its local experts are then gathered from that copy.  One tile per
            // 64-token routing block, taken by whoever comes first.
            while (ok) {
                int blk = 0;
                if (lane == 0) blk = (int)atomicAdd(&S.cs->q_pull, 1u);
                blk = __shfl_sync(0xffffffffu, blk, 0);
                if (blk >= p.nblk) break;
                const unsigned long long um = lmask ? lmask[blk * (kMaxEE + 1) + kMaxEE] : __ldcg(p.uniq_mask + blk);
                const int n = __popcll(um);
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const int bit = lane + 32 * hh;
                    if ((um >> bit) & 1ull) M.tok[__popcll(um & ((1ull << bit) - 1ull))] = blk * kRouteBlock + bit;
                }
                __syncwarp();
                if (lane == 0) {
                    if (n == 0) {
                        red_release_add_u32(&S.cs->pull_done, 1u);
                    } else {
                        const int Rp = min(R, 32);
                        for (int r0 = 0; r0 < n; r0 += Rp) {
                            const int nr = min(Rp, n - r0);
                            if (!mbar_wait(&S.dv_empty[b], ph ^ 1u, p, 14)) { ok = false; break; }
                            M.mv[b].a = 0; M.mv[b].b = nr; M.mv[b].c = blk; M.mv[b].d = (r0 + nr >= n) ? 4 : 3;
                            for (int i = 0; i < nr; ++i) M.mv[b].tok[i] = M.tok[r0 + i];
                            mbar_arrive_expect_tx(&S.dv_full[b], (uint32_t)nr * rowb);
                            const uint32_t dst = smem_u32(stages + b * kMvBuf);
                            for (int i = 0; i < nr; ++i)
                                bulk_load(dst + (uint32_t)i * rowb, p.x + (size_t)M.tok[r0 + i] * p.H, rowb, &S.dv_full[b]);
                            if (++b == kStages) { b = 0; ph ^= 1u; }
                        }
                    }
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                __syncwarp();
            }
            // rows may be gathered from xs only when every block has been staged: have the storer
            // complete and publish what it still holds back (d = 5), then wait for everybody's blocks
            if (lane == 0 && ok) {
                if (mbar_wait(&S.dv_empty[b], ph ^ 1u, p, 16)) {
                    M.mv[b].d = 5;
                    mbar_arrive(&S.dv_full[b]);
                    if (++b == kStages) { b = 0; ph ^= 1u; }
                } else ok = false;
            }
            if (lane == 0 && ok && max_tiles > 0) ok = flag_wait_ge(&S.cs->pull_done, (unsigned)p.nblk, p, 15);
            ok = __shfl_sync(0xffffffffu, ok, 0);
            // only lane 0 walked the ring so far; from here on every lane addresses the buffers
            b = __shfl_sync(0xffffffffu, b, 0);
            ph = __shfl_sync(0xffffffffu, ph, 0);
        }
        for (int taken = 0; ok && taken < max_tiles; ++taken) {
            int mb = (int)blockIdx.x;
            if (taken > 0) {
                if (lane == 0) mb = n_disp + (int)atomicAdd(&S.cs->q_disp, 1u);
                mb = __shfl_sync(0xffffffffu, mb, 0);
            }
            if (mb >= S.nmb) { if (taken > 0) break; else continue; }
            int row0, nrows, seg;
            decode_mblock(S, p.EE, mb, row0, nrows, seg);
            if (lmask == nullptr) {
                for (int i = lane; i < nrows; i += 32) M.tok[i] = __ldcg(p.token_of + row0 + i);
            } else {
                // row r of expert e = the r-th token that selected it, in token order; a shared expert's
                // row r is token r
                const int e = seg % p.EE;
                for (int i = lane; i < nrows; i += 32) {
                    int rank = row0 + i - S.offsets[e];
                    int tok = rank;
                    if (e < p.E) {
                        tok = 0;
                        for (int bb = 0; bb < p.nblk; ++bb) {
                            const unsigned long long mk = lmask[bb * (kMaxEE + 1) + e];
                            const int c = __popcll(mk);
                            if (rank < c) { tok = bb * kRouteBlock + nth_set_bit(mk, rank); break; }
                            rank -= c;
                        }
                    }
                    M.tok[i] = tok;
                }
            }
            __syncwarp();
            for (int r0 = 0; r0 < nrows && ok; r0 += R) {
                const int nr = min(R, nrows - r0);
                if (lane == 0) {
                    if (!mbar_wait(&S.dv_empty[b], ph ^ 1u, p, 11)) ok = false;
                    else {
                        M.mv[b].a = row0 + r0; M.mv[b].b = nr; M.mv[b].c = mb; M.mv[b].d = (r0 + nr >= nrows) ? 1 : 0;
                        mbar_arrive_expect_tx(&S.dv_full[b], (uint32_t)nr * rowb);
                    }
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                // the expected byte count is registered; the lanes issue the row copies side by side
                const uint32_t dst = smem_u32(stages + b * kMvBuf);
                for (int i = lane; i < nr; i += 32) {
                    const int tk = M.tok[r0 + i];
                    // a remote token (another rank's shard) is read from its staged copy
                    const __nv_bfloat16 *src = (p.ep_size > 1 && tk / p.ep_tshard != p.ep_rank) ? p.xs : p.x;
                    bulk_load(dst + (uint32_t)i * rowb, src + (size_t)tk * p.H, rowb, &S.dv_full[b]);
                }
                if (++b == kStages) { b = 0; ph ^= 1u; }
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            __syncwarp();
        }
        if (lane == 0 && ok && mbar_wait(&S.dv_empty[b], ph ^ 1u, p, 12)) {
            M.mv[b].d = 2;
            mbar_arrive(&S.dv_full[b]);
        }
        // a wait gave up (or the abort word was seen): copies this warp issued may still be landing in
        // this CTA's buffers; let them land before the CTA can leave
        if (!ok && lane == 0) linger_after_abort();
        __syncwarp();
    } else if (warp == 1) {
        // ---- storer: one bulk store per buffer.  A buffer is handed back as soon as the store has
        // read it; an m-block's flag is published once the stores up to its last one have completed
        // (checked with a lag of kFlagLag stores, so the copy engine never drains).
        if (lane == 0) {
            constexpr int kFlagLag = 4, kPend = 8;
            int b = 0, n = 0;
            uint32_t ph = 0;
            int prev_buf = -1;
            int pe_idx[kPend], pe_mb[kPend], pe_rows[kPend];      // tile ends not yet published (mb < 0: a staged block)
            unsigned long long pe_t0[kPend];
            for (int i = 0; i < kPend; ++i) { pe_idx[i] = 0; pe_mb[i] = 0; pe_rows[i] = 0; pe_t0[i] = 0ull; }
            int pe_head = 0, pe_tail = 0;
            auto publish_upto = [&](int done_idx) {      // stores with index <= done_idx have completed
                bool fenced = false;
                while (pe_head != pe_tail && pe_idx[pe_head % kPend] <= done_idx) {
                    const int s8 = pe_head % kPend;
                    // (the bulk stores have completed; the release below orders them for whoever acquires the flag)
                    if (!fenced) { fence_proxy_async_global(); fenced = true; }
                    if (pe_mb[s8] < 0) {
                        red_release_add_u32(&S.cs->pull_done, 1u);      // a block of remote tokens is staged
                    } else {
                        if (pe_mb[s8] != p.withhold_mb) {      // the m-block's rows count in on the row tiles they are part of
                            int row0, nrows, seg;
                            decode_mblock(S, p.EE, pe_mb[s8], row0, nrows, seg);
                            const int rows = S.seg_rows[seg], pts = S.seg_pt0[seg + 1] - S.seg_pt0[seg], rel = row0 - S.seg_row0[seg];
                            for (int i = rowtile_of_rel(rows, pts, rel); i < pts; ++i) {
                                int first, n;
                                rowtile_span(rows, pts, i, first, n);
                                if (first >= rel + nrows) break;
                                red_release_add_u32(&S.xe_ready[S.seg_pt0[seg] + i], (unsigned)(min(first + n, rel + nrows) - max(first, rel)));
                            }
                        }
                        trace_ev(p, S, kEvDispatch, (unsigned)pe_mb[s8], pe_t0[s8], trace_now(p), (unsigned)pe_rows[s8]);
                    }
                    ++pe_head;
                }
            };
            unsigned long long tile_t0 = trace_now(p);
            for (;;) {
                if (!mbar_wait(&S.dv_full[b], ph, p, 13)) break;
                const int da = M.mv[b].a, db = M.mv[b].b, dc = M.mv[b].c, dd = M.mv[b].d;
                if (dd == 2) break;
                if (dd == 5) {      // flush: everything stored so far becomes visible and is published
                    bulk_wait<0>();
                    if (prev_buf >= 0) { mbar_arrive(&S.dv_empty[prev_buf]); prev_buf = -1; }
                    publish_upto(n);
                    mbar_arrive(&S.dv_empty[b]);
                    if (++b == kStages) { b = 0; ph ^= 1u; }
                    continue;
                }
                if (dd >= 3) {      // staged remote tokens: one store per row, to the token's own slot of xs
                    for (int i = 0; i < db; ++i)
                        bulk_store(p.xs + (size_t)M.mv[b].tok[i] * p.H, smem_u32(stages + b * kMvBuf) + (uint32_t)i * rowb, rowb);
                } else {
                    bulk_store(p.xe + (size_t)da * p.H, smem_u32(stages + b * kMvBuf), (uint32_t)db * rowb);
                }
                bulk_commit();
                if (prev_buf >= 0) { bulk_wait_read<1>(); mbar_arrive(&S.dv_empty[prev_buf]); }
                prev_buf = b;
                if (dd == 1 || dd == 4) {
                    if (pe_tail - pe_head == kPend) { bulk_wait<0>(); publish_upto(n); }
                    const int s8 = pe_tail % kPend;
                    pe_idx[s8] = n; pe_mb[s8] = dd == 4 ? -1 : dc; pe_rows[s8] = db; pe_t0[s8] = tile_t0;
                    ++pe_tail;
                    tile_t0 = trace_now(p);
                }
                if (n >= kFlagLag && pe_head != pe_tail) { bulk_wait<kFlagLag>(); publish_upto(n - kFlagLag); }
                ++n;
                if (++b == kStages) { b = 0; ph ^= 1u; }
            }
            bulk_wait<0>();
            if (prev_buf >= 0) mbar_arrive(&S.dv_empty[prev_buf]);
            publish_upto(n);
        }
        __syncwarp();
    }
    __syncthreads();
}

// The dispatch in token order, for the plans in which every CTA dispatches and nothing is staged: a token's row of x is
// read once and written to its k + S rows of Xe.  (In m-block order every row was read for each of its experts, from HBM
// where x does not fit L2, an m-block's 128 rows were one SM's chain of copies, and nothing began before the
// permutation of ALL tokens was final.)  The row tiles' ready flags count their rows in.
// (test hook) does row tile rt have rows of the withheld m-block?
__device__ __noinline__ bool withheld(int mb, int EE, int rt)
{
    const SmemTail &S = smem_tail();
    if (mb >= S.nmb) return false;
    int row0, nrows, seg;
    decode_mblock(S, EE, mb, row0, nrows, seg);
    const int rows = S.seg_rows[seg], pts = S.seg_pt0[seg + 1] - S.seg_pt0[seg], rel = row0 - S.seg_row0[seg], i = rt - S.seg_pt0[seg];
    return i >= rowtile_of_rel(rows, pts, rel) && i <= rowtile_of_rel(rows, pts, rel + nrows - 1);
}
__device__ __forceinline__ void publish_row(const KParams &p, SmemTail &S, int rt, unsigned long long t0)
{
    if (p.withhold_mb >= 0 && withheld(p.withhold_mb, p.EE, rt)) return;
    if (p.trace == nullptr) {
        red_release_add_u32(&S.xe_ready[rt], 1u);
    } else {      // the timeline has one record per m-block, made by whoever completes its row tile
        const unsigned before = atom_acqrel_add_u32(&S.xe_ready[rt], 1u);
        int lo = 0, hi = p.EE;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (S.seg_pt0[mid] <= rt) lo = mid; else hi = mid;
        }
        const int i = rt - S.seg_pt0[lo], mb = S.seg_mb0[lo] + 2 * i;
        int first, n;
        rowtile_span(S.seg_rows[lo], S.seg_pt0[lo + 1] - S.seg_pt0[lo], i, first, n);
        if ((int)before + 1 == n) {
            trace_ev(p, S, kEvDispatch, (unsigned)mb, t0, trace_now(p), (unsigned)n);
            if (mb + 1 < S.seg_mb0[lo + 1]) trace_ev(p, S, kEvDispatch, (unsigned)(mb + 1), t0, trace_now(p), 0u);
        }
    }
}
__device__ __forceinline__ int rowtile_of(const SmemTail &S, int row, int e)      // K = 1: segment = expert
{
    return S.seg_pt0[e] + rowtile_of_rel(S.seg_rows[e], S.seg_pt0[e + 1] - S.seg_pt0[e], row - S.seg_row0[e]);
}

// Small batches (a few tokens per CTA): warps that have no work yet when the GEMM phase begins - the releasing warp and
// the epilogue warps, wid = 0..kInlineWarps-1 - copy the rows with ordinary loads and stores, while the producers
// already fetch the first tiles' weights.  Nothing stands in front of the GEMM phase then (8 experts, T = 256: 39.2 ->
// 35.2 us; DSv2-Lite-shaped, T = 256: 214.3 -> 211.2; Qwen3.5-35B-shaped, T = 1023: 315.7 -> 310.2).
//   one routing block (T <= 64, every CTA has all masks): unit = a token and a share of its experts, spread over all CTAs;
//   otherwise: this CTA's own routing block, whose rows it placed itself.
constexpr int kInlineWarps = 5;
__device__ __forceinline__ void dispatch_inline(const KParams &p, SmemTail &S, uint8_t *stages, int wid)
{
    const int lane = threadIdx.x & 31, kk = p.k + p.S, n_sm = (int)gridDim.x;
    const unsigned long long td0 = trace_now(p);
    const bool local = p.nblk <= kLocalBlocks;
    const unsigned long long *mask = reinterpret_cast<const unsigned long long *>(stages + kStages * kStageBytes);
    const int parts = local ? max(1, min(kk, n_sm * kInlineWarps / p.T)) : 1;
    const int unit0 = local ? (int)blockIdx.x * kInlineWarps + wid : wid;
    const int units = local ? p.T * parts : 1 << p.lg_rb, step = local ? n_sm * kInlineWarps : kInlineWarps;
    for (int w = unit0; w < units; w += step) {
        const int t = local ? w % p.T : ((int)blockIdx.x << p.lg_rb) + w, part = local ? w / p.T : 0;
        if (t >= p.T) break;
        int n = 0, row = 0, rt = 0;      // lane i: the i-th destination of this unit and its row tile
        if (local) {
            int seen = 0;
            for (int e0 = 0; e0 < p.EE; e0 += 32) {
                const int e = e0 + lane;
                unsigned all = __ballot_sync(0xffffffffu, e < p.EE && (e >= p.E || ((mask[e] >> t) & 1ull)));
                for (; all; all &= all - 1u, ++seen) {
                    if (seen % parts != part) continue;
                    const int es = e0 + __ffs((int)all) - 1;
                    if (lane == n) {
                        row = S.offsets[es] + (es < p.E ? __popcll(mask[es] & ((1ull << t) - 1ull)) : t);
                        rt = rowtile_of(S, row, es);
                    }
                    ++n;
                }
            }
        } else {
            n = kk;
            if (lane < p.k) {
                const size_t at = (size_t)t * p.k + lane;
                row = __ldcg(p.row_of + at);
                rt = rowtile_of(S, row, __ldcg(p.topk_idx + at));
            } else if (lane < kk) {
                row = S.offsets[p.E + lane - p.k] + t;
                rt = rowtile_of(S, row, p.E + lane - p.k);
            }
        }
        const uint4 *src = reinterpret_cast<const uint4 *>(p.x + (size_t)t * p.H);
        const int vecs = p.H >> 3;      // a multiple of 16
        for (int v0 = 0; v0 < vecs; v0 += 128) {
            uint4 q[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (v0 + 32 * i + lane < vecs) q[i] = __ldg(src + v0 + 32 * i + lane);
            for (int j = 0; j < n; ++j) {
                uint4 *dst = reinterpret_cast<uint4 *>(p.xe + (size_t)__shfl_sync(0xffffffffu, row, j) * p.H);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (v0 + 32 * i + lane < vecs) dst[v0 + 32 * i + lane] = q[i];
            }
        }
        __syncwarp();      // the rows are written; the release below is cumulative
        if (lane < n) {
            fence_proxy_async_global();      // (TMA reads them)
            publish_row(p, S, rt, td0);
        }
    }
    __syncwarp();
}

// Large batches, 16-token tiles from the queue: bulk loads bring as many tokens as fit a 32 KB ring buffer (they are
// neighbours in x: one copy); the lanes of the storing warp write each row out with one bulk store per destination and
// publish it once those stores have completed, two buffers later.  Bound by HBM writes; T = 16384, H = 4096, k = 8:
// 310 -> 230 us.
__device__ __forceinline__ void dispatch_tokens(const KParams &p, SmemTail &S, uint8_t *stages)
{
    TokScratch &M = *reinterpret_cast<TokScratch *>(stages + kStages * kStageBytes + kEpiStageBytes / 2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n_sm = (int)gridDim.x;
    fence_proxy_async_shared();      // the buffers held routing scratch written with ordinary stores
    __syncthreads();
    const uint32_t rowb = (uint32_t)p.H * 2u;
    const int kk = p.k + p.S;
    const int per_buf = min(kMvBuf / (int)rowb, kTokEnt / kk);      // tokens per buffer (at least 1: H <= 16384, kk <= 24)
    if (warp == 0) {
        // ---- loader
        int b = 0;
        uint32_t ph = 0;
        bool ok = true;
        if (lane == 0) ok = flag_wait_ge(&S.cs->fix_done, (unsigned)p.nrb, p, 10);
        ok = __shfl_sync(0xffffffffu, ok, 0);
        const int ntile = (p.T + 15) / 16;
        for (int q = (int)blockIdx.x; ok && q < ntile;) {
            const int t1 = min(p.T, q * 16 + 16);
            for (int t = q * 16; t < t1; t += per_buf) {
                const int nt = min(per_buf, t1 - t), n = nt * kk;
                ok = __all_sync(0xffffffffu, mbar_wait(&S.dv_empty[b], ph ^ 1u, p, 11));
                if (!ok) break;
                for (int i = lane; i < n; i += 32) {
                    const int tt = i / kk, j = i - tt * kk;
                    const size_t at = (size_t)(t + tt) * p.k + j;
                    const int row = j < p.k ? __ldcg(p.row_of + at) : S.offsets[p.E + j - p.k] + t + tt;
                    M.row[b][i] = row;
                    M.rt[b][i] = rowtile_of(S, row, j < p.k ? __ldcg(p.topk_idx + at) : p.E + j - p.k);
                }
                __syncwarp();
                if (lane == 0) {
                    M.n[b] = n;
                    mbar_arrive_expect_tx(&S.dv_full[b], (uint32_t)nt * rowb);
                    bulk_load(smem_u32(stages + b * kMvBuf), p.x + (size_t)t * p.H, (uint32_t)nt * rowb, &S.dv_full[b]);
                }
                if (++b == kStages) { b = 0; ph ^= 1u; }
            }
            if (lane == 0) q = n_sm + (int)atomicAdd(&S.cs->q_disp, 1u);
            q = __shfl_sync(0xffffffffu, q, 0);
        }
        if (ok && __all_sync(0xffffffffu, mbar_wait(&S.dv_empty[b], ph ^ 1u, p, 12))) {
            if (lane == 0) { M.n[b] = -1; mbar_arrive(&S.dv_full[b]); }
        } else if (lane == 0) linger_after_abort();      // copies of this warp may still be landing in this CTA's buffers
        __syncwarp();
    } else if (warp == 1) {
        // ---- storer
        constexpr int kLag = 2;
        int b = 0, n_buf = 0;
        uint32_t ph = 0;
        const unsigned long long td0 = trace_now(p);
        auto publish = [&](int buf) {      // the stores out of `buf` have completed
            fence_proxy_async_global();
            const int n = M.n[buf];
            for (int i = lane; i < n; i += 32) publish_row(p, S, M.rt[buf][i], td0);
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.dv_empty[buf]);
        };
        bool ok = true;
        for (;;) {
            ok = __all_sync(0xffffffffu, mbar_wait(&S.dv_full[b], ph, p, 13));
            if (!ok) break;
            const int n = M.n[b];
            if (n < 0) break;
            const uint32_t src = smem_u32(stages + b * kMvBuf);
            for (int i = lane; i < n; i += 32)
                bulk_store(p.xe + (size_t)M.row[b][i] * p.H, src + (uint32_t)(i / kk) * rowb, rowb);
            bulk_commit();
            if (n_buf >= kLag) { bulk_wait<kLag>(); publish(b >= kLag ? b - kLag : b + kStages - kLag); }
            ++n_buf;
            if (++b == kStages) { b = 0; ph ^= 1u; }
        }
        bulk_wait<0>();
        __syncwarp();
        if (ok)
            for (int i = min(n_buf, kLag); i > 0; --i) publish(b >= i ? b - i : b + kStages - i);
    }
    __syncthreads();
}

// ------------------------------------------------------------------------------------ phase C: combine

// Tile = 16 tokens.  out[t] = sum_j gate[t,j] * y[row_of[t,j]] in slot order, then the shared
// experts with weight 1; fp32 accumulate, bf16 store.  Warp 0 gathers, per token and per piece of
// W columns, the k+S source rows with bulk loads into a ring of 32 KB buffers; warps 2..7 reduce
// each full buffer from shared memory and write the output row piece with coalesced stores.
__device__ __forceinline__ void combine_phase(const KParams &p, SmemTail &S, uint8_t *stages)
{
    MoveScratch &M = move_scratch(stages);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    fence_proxy_async_shared();
    __syncthreads();
    const int kk = p.k + p.S;
    const int W = min(p.H, ((kMvBuf / (2 * kk)) / 64) * 64);     // columns per piece (128-byte multiple)
    const int g = kFine / S.K;
    if (warp == 0) {
        // ---- loader
        int b = 0;
        uint32_t ph = 0;
        int ready_upto = -1;     // chunks [0, ready_upto] are known complete
        bool perm_final = false; // the permutation's rows (row_of, gates) are known final
        bool ok = true;
        for (;;) {
            int q = 0;
            if (lane == 0) q = (int)atomicAdd(&S.cs->q_comb, 1u);
            q = __shfl_sync(0xffffffffu, q, 0);
            if (q >= S.n_comb) break;
            const int t0 = q * S.comb_tok;
            const int chunk = (((t0 / kRouteBlock) * kFine) / p.nblk) / g;
            const int ntok = min(S.comb_tok, p.T - t0);
            // the tile's rows and gates are final once the permutation is; they are fetched before the wait for
            // the chunk's last GEMM tile, so that only the row copies themselves follow that wait
            if (!perm_final) {
                if (lane == 0) ok = flag_wait_ge(&S.cs->fix_done, (unsigned)p.nrb, p, 20);
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                perm_final = true;
            }
            for (int i = lane; i < ntok * kk; i += 32) {
                const int tt = i / kk, j = i - tt * kk, t = t0 + tt;
                M.crow[tt][j] = j < p.k ? __ldcg(p.row_of + (size_t)t * p.k + j) : S.offsets[p.E + (j - p.k)] + t;
                M.cgate[tt][j] = j < p.k ? __ldcg(p.gates + (size_t)t * p.k + j) : 1.0f;
            }
            __syncwarp();
            if (chunk > ready_upto) {
                if (lane == 0) {
                    const unsigned long long tw0 = trace_now(p);
                    for (int j = ready_upto + 1; ok && j <= chunk; ++j) {
                        ok = flag_wait_ge(&S.cs->y_done[j], y_done_target(S, p, j), p, 21);
                    }
                    trace_ev(p, S, kEvWaitChunk, (unsigned)chunk, tw0, trace_now(p), 0u);
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                ready_upto = chunk;
            }
            const unsigned long long tc0 = trace_now(p);
            for (int tt = 0; tt < ntok && ok; ++tt) {
                // lane j owns slot j of the token: its rank among the slots that have a row here (slots
                // whose expert lives on another rank have row -1 and are skipped)
                const int myrow = lane < kk ? M.crow[tt][lane] : -1;
                const unsigned vmask = __ballot_sync(0xffffffffu, myrow >= 0);
                const int nv = __popc(vmask), mypos = __popc(vmask & ((1u << lane) - 1u));
                // a token with few rows here (expert-parallel share) takes wider pieces: as many columns
                // as fit the buffer with the rows it really has
                const int Wt = nv >= kk ? W : min(p.H, ((kMvBuf / (2 * max(nv, 1))) / 64) * 64);
                for (int col0 = 0; col0 < p.H && ok; col0 += Wt) {
                    const int w = min(Wt, p.H - col0);
                    if (lane == 0) {
                        if (!mbar_wait(&S.cb_empty[b], ph ^ 1u, p, 22)) ok = false;
                        else {
                            M.mv[b].a = t0 + tt; M.mv[b].b = col0; M.mv[b].c = w; M.mv[b].d = 0; M.mv[b].n = nv;
                        }
                    }
                    ok = __shfl_sync(0xffffffffu, ok, 0);
                    if (!ok) break;
                    if (myrow >= 0) M.mv[b].g[mypos] = M.cgate[tt][lane];
                    __syncwarp();
                    if (lane == 0) {
                        if (nv > 0) mbar_arrive_expect_tx(&S.cb_full[b], (uint32_t)(nv * w * 2));
                        else mbar_arrive(&S.cb_full[b]);
                    }
                    __syncwarp();
                    // the byte count is registered; the lanes issue the row copies side by side
                    if (myrow >= 0)
                        bulk_load(smem_u32(stages + b * kMvBuf) + (uint32_t)(mypos * w * 2),
                                  p.y + (size_t)myrow * p.H + col0, (uint32_t)(w * 2), &S.cb_full[b]);
                    if (++b == kStages) { b = 0; ph ^= 1u; }
                }
            }
            if (lane == 0) trace_ev(p, S, kEvCombine, (unsigned)q, tc0, trace_now(p), 0u);
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            __syncwarp();
        }
        if (lane == 0 && ok && mbar_wait(&S.cb_empty[b], ph ^ 1u, p, 23)) {
            M.mv[b].d = 2;
            mbar_arrive(&S.cb_full[b]);
        }
        if (!ok && lane == 0) linger_after_abort();      // as in the dispatch loader
        __syncwarp();
    } else if (warp >= 2) {
        // ---- reducers
        const int ctid = tid - 64;
        int b = 0;
        uint32_t ph = 0;
        for (;;) {
            bool ok = mbar_wait(&S.cb_full[b], ph, p, 24);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const MvDesc &d = M.mv[b];
            if (d.d == 2) break;
            const int w = d.c, nv = w >> 3, nrow = d.n;
            const uint32_t src = smem_u32(stages + b * kMvBuf);
            __nv_bfloat16 *dst = p.out + (size_t)d.a * p.H + d.b;
            for (int v = ctid; v < nv; v += kCombWarps * 32) {
                float a0[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) a0[i] = 0.f;
                for (int j = 0; j < nrow; ++j) {
                    const uint4 q4 = ld_shared_v4(src + (uint32_t)(j * w * 2 + v * 16));
                    const float gw = d.g[j];
                    a0[0] = fmaf(gw, bf16lo_to_f32(q4.x), a0[0]); a0[1] = fmaf(gw, bf16hi_to_f32(q4.x), a0[1]);
                    a0[2] = fmaf(gw, bf16lo_to_f32(q4.y), a0[2]); a0[3] = fmaf(gw, bf16hi_to_f32(q4.y), a0[3]);
                    a0[4] = fmaf(gw, bf16lo_to_f32(q4.z), a0[4]); a0[5] = fmaf(gw, bf16hi_to_f32(q4.z), a0[5]);
                    a0[6] = fmaf(gw, bf16lo_to_f32(q4.w), a0[6]); a0[7] = fmaf(gw, bf16hi_to_f32(q4.w), a0[7]);
                }
                st_cs_v4(dst + v * 8, make_uint4(pack_bf16x2(a0[0], a0[1]), pack_bf16x2(a0[2], a0[3]),
                                                 pack_bf16x2(a0[4], a0[5]), pack_bf16x2(a0[6], a0[7])));
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.cb_empty[b]);
            if (++b == kStages) { b = 0; ph ^= 1u; }
        }
    }
    __syncthreads();
}

// ------------------------------------------------------------------------------------ phase B: GEMM

// Tensor maps of the GEMM operands: bf16 matrices, boxes of 64 columns (one 128-byte swizzle row) by
// 128 rows (64 rows for the gate and up halves of a swapped tile's weight operand; 8, 16, 32 or 64 rows for its row
// operand, whichever covers each CTA's half of the tile's rows, or what is left of it behind a first box of 64).
// x: the input itself, boxes of half the batch's tokens rounded up to 8 or 16 (only where KParams::direct is set).
struct TmaMaps { CUtensorMap xe, wgu, h, wd, wgu64, xe_n[4], h_n[4], x; };

struct PipeState {     // per-role ring positions; they persist across the tiles of a phase
    int stage = 0;  uint32_t stage_phase = 0;
    int acc = 0;    uint32_t acc_phase = 0;
    int slot = 0;   uint32_t slot_phase = 0;
    __device__ __forceinline__ void next_stage() { if (++stage == kStages) { stage = 0; stage_phase ^= 1u; } }
    __device__ __forceinline__ void next_acc() { if (++acc == 2) { acc = 0; acc_phase ^= 1u; } }
    __device__ __forceinline__ void next_slot() { if (++slot == kTinfo) { slot = 0; slot_phase ^= 1u; } }
    int rel = 0;    uint32_t rel_phase = 0;
    __device__ __forceinline__ void next_rel() { if (++rel == kRel) { rel = 0; rel_phase ^= 1u; } }
};

__device__ __forceinline__ float silu_mul(float g, float u)
{
    return __fdividef(g, 1.0f + __expf(-g)) * u;
}

// A consumer of the tile-descriptor ring hands its slot back with a barrier arrival, after which the
// scheduler (for the peer CTA: a thread of ANOTHER CTA, through remote stores) may overwrite the slot.
// The copy of the descriptor must have LANDED in this thread's registers by then.  Program order alone
// does not say so: the arrival has CTA scope (a cluster-scope release would wait for the thread's
// global stores, ~1000 cycles) and no instruction reads the loaded words before it is issued, so the
// shared-memory loads can still be in flight when the slot is rewritten.  Storing a fold of all eight
// words to a scratch word makes the hardware wait for them here: a store cannot issue before its
// operand has arrived, and the arrival is issued after the store.  (An empty asm statement that
// merely names the words generates no instruction and therefore no wait.)
// Seen without it, about once in 300 000 launches and only in the peer CTA: warps reading different
// row counts for one swapped tile, the up/gate exchange of its epilogue running out of step, the
// accumulator never handed back, a bounded wait running out.
__device__ __forceinline__ void tile_info_landed(const TileInfo &ti, int *scratch)
{
    *reinterpret_cast<volatile int *>(scratch) = ti.type ^ ti.mb ^ ti.rt ^ ti.row0 ^ ti.nrows ^ ti.e ^ ti.n ^ ti.chunk ^ ti.nkb;
}

// bounded wait on a barrier whose guarded data may come from the peer CTA
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t *bar, uint32_t parity, const KParams &p, int where)
{
    if (mbar_try_wait_cluster(bar, parity)) return true;
    unsigned long long t0 = 0;
    unsigned it = 0;
    unsigned ab = 0u;      // looked at one round late, see mbar_wait
    while (!mbar_try_wait_cluster(bar, parity)) {
        if ((++it & 31u) == 0u) {
            if (ab) { note_failed_wait(p.wait_log, where, smem_u32(bar), parity, 2); return false; }
            ab = ld_relaxed_u32(&smem_tail().cs->abort);
            const unsigned long long now = globaltimer_ns();
            if (t0 == 0) t0 = now;
            else if ((long long)(now - t0) > (long long)p.timeout_ns) {
                give_up(p.ctl, where);
                note_failed_wait(p.wait_log, where, smem_u32(bar), parity, 1);
                return false;
            }
        }
    }
    return true;
}

// 32 rows x 32 columns of bf16 held one row per thread (16 packed words each) go out through the
// warp's own 2 KB of shared memory, so that every store instruction writes 16 rows x 64 contiguous
// bytes (two lanes per row) instead of 32 rows x 32 bytes.  An SM retires st.global at 32 B per
// cycle but at most one 128-byte line every two cycles: one row per thread is 15.8 B/clk per SM,
// two lanes per row 31 B/clk (measured with a store-only probe, alone or on all SMs).
// Shared-memory layout: row r at r*64, its 16-byte chunk c at position c ^ ((r >> 1) & 3): the
// row-per-thread writes and the two-lanes-per-row reads are both free of bank conflicts.
// dst = first of the warp's 32 rows (this batch's first column), pitch in elements.
__device__ __forceinline__ void staged_store_32(const uint32_t (&o)[16], uint32_t stage, __nv_bfloat16 *dst, int pitch,
                                                int rows_valid, int lane)
{
    const uint32_t wbase = stage + (uint32_t)lane * 64u, wsw = (uint32_t)((lane >> 1) & 3);
#pragma unroll
    for (int c = 0; c < 4; ++c)
        st_shared_v4(wbase + (((uint32_t)c ^ wsw) << 4), make_uint4(o[4 * c], o[4 * c + 1], o[4 * c + 2], o[4 * c + 3]));
    __syncwarp();
    const int half = lane & 1;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int r = 16 * j + (lane >> 1);
        const uint32_t rbase = stage + (uint32_t)r * 64u, rsw = (uint32_t)((r >> 1) & 3);
        const uint4 q0 = ld_shared_v4(rbase + (((uint32_t)(2 * half) ^ rsw) << 4));
        const uint4 q1 = ld_shared_v4(rbase + (((uint32_t)(2 * half + 1) ^ rsw) << 4));
        if (r < rows_valid) {
            const uint32_t v[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
            st_v8(dst + (size_t)r * pitch + half * 16, v);
        }
    }
    __syncwarp();      // the region is rewritten by the next batch
}

// S.budget = how many pair tiles this CTA pair may claim (the steal count for a movement pair); S.direct: the
// gate/up tiles take the batch's tokens themselves as their row operand (all tiles are swapped ones then).  They and
// the other scalars come through shared memory: the epilogue has no registers to spare for values that live across it.
__device__ __forceinline__ void gemm_phase(const KParams &p, SmemTail &S, uint8_t *stages, const TmaMaps *tm)
{
    PipeState ps;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_ctarank();      // 0 = leader (issues the MMAs), 1 = peer
    fence_proxy_async_shared();     // the stage buffers were last touched by ordinary stores (routing scratch)
    __syncthreads();

    if (S.inline_disp && warp >= 8 - kInlineWarps) {
        dispatch_inline(p, S, stages, warp - (8 - kInlineWarps));
        // Its warps look rows up in the routing masks, and a swapped gate/up tile of more than 32 rows trades values where
        // the masks are (lower exchange buffers): no warp goes on to its epilogue before the others are done with them.
        // No barrier (inline_disp = 1) where the batch has at most 32 tokens, whose tiles use the upper buffers only, or more
        // than one routing block, whose rows are not looked up in masks.
        if (S.inline_disp > 1) named_barrier_sync<1, kInlineWarps * 32>();
    }

    if (warp == 2 && rank == 0) {
        // ---------------- scheduler (leader only): claims pair tiles in queue order, waits until their
        // inputs are ready, then publishes the tile to both CTAs' descriptor rings.  Runs up to
        // kTinfo tiles ahead of the MMAs, so claim and flag latencies stay off the critical path.
        if (lane == 0) {
            int taken = 0;
            // this die's list first; when it has run out, the other one's.  A tile waits only for tiles before it in
            // its own list and for the dispatch, so of all claimed tiles the one claimed first can always proceed.
            const int per_pt = p.nt0 + p.nt1;
            const int n_list0 = S.K == 1 ? S.split_pt * per_pt : S.n_gemm;
            int list = n_list0 == S.n_gemm ? 0 : S.die;
            bool second = false;
            auto claim = [&]() -> int {
                for (;;) {
                    const int c = (int)atomicAdd(&S.cs->q_gemm[list], 1u);
                    if (c < (list ? S.n_gemm - n_list0 : n_list0)) return c;
                    if (second) return 0x7fffffff;
                    second = true;
                    list ^= 1;
                }
            };
            int g_next = (S.budget > 0 || S.elastic) ? claim() : 0x7fffffff;
            for (;;) {
                const int g = g_next;
                const unsigned long long tp0 = trace_now(p);
                TileInfo tl, tp;
                if (g >= S.n_gemm) { tl.type = tp.type = 2; tl.mb = tp.mb = -1; tl.nrows = tp.nrows = 0; tl.chunk = tp.chunk = 0; }
                else decode_pair_tile(S, p, list, g, tl, tp);
                // Are the tile's rows there?  If not, it is handed over all the same: the producers fetch the weights of its
                // first k-steps meanwhile (8 experts, T = 256: 41.4 -> 39.2 us).
                const bool g0 = tl.type == 0 || tl.type == 3;
                const unsigned *fl = tl.type == 2 ? nullptr : (g0 ? S.xe_ready : S.h_ready) + tl.rt;
                const unsigned need = g0 ? (unsigned)(tl.type == 0 ? kBM + tp.nrows : tl.nrows) : (unsigned)(p.nt0 * 2 * kEpiWarps);
                const bool waits = tl.type != 2 && !(S.direct && tl.type == 3);      // (x was there before the launch)
                const bool late = waits && ld_acquire_u32(fl) < need;
                if (late) { tl.chunk |= kTileLate; tp.chunk |= kTileLate; }
                if (!mbar_wait(&S.ti_empty[ps.slot], ps.slot_phase ^ 1u, p, 30)) break;
                S.ti[ps.slot] = tl;
                {
                    const uint32_t dst = mapa_u32(smem_u32(&S.ti[ps.slot]), 1u);
                    const uint32_t *src = reinterpret_cast<const uint32_t *>(&tp);
#pragma unroll
                    for (int w = 0; w < (int)(sizeof(TileInfo) / 4); ++w) st_cluster_u32(dst + 4 * w, src[w]);
                }
                // the tile's input rows may have been written with ordinary stores on other SMs and are read by TMA
                // next: the cross-proxy fence sits here, after the acquire and before the hand-over to the
                // producers, off their critical path
                if (waits && !late) fence_proxy_async_global();
                mbar_arrive(&S.ti_full[ps.slot]);
                mbar_arrive_cluster(mapa_u32(smem_u32(&S.ti_full[ps.slot]), 1u));
                if (late) {
                    if (!flag_wait_ge(fl, need, p, g0 ? 31 : 32)) break;
                    fence_proxy_async_global();
                    mbar_arrive(&S.ti_late[ps.slot]);
                    mbar_arrive_cluster(mapa_u32(smem_u32(&S.ti_late[ps.slot]), 1u));
                }
                if (p.trace && tl.type != 2)      // (the id is the tile's place in the whole queue, the second list behind the first)
                    trace_ev(p, S, kEvGemmLoad, (unsigned)(list ? S.split_pt * per_pt + g : g), tp0, trace_now(p), 0u);
                ps.next_slot();
                if (tl.type == 2) break;
                // the next claim's round trip comes after the hand-over
                ++taken;
                bool more = taken < S.budget;
                if (!more && S.elastic) {
                    // the steal quota is used up: keep taking GEMM tiles for as long as the next
                    // combine chunk has not been produced yet (nothing else to do meanwhile)
                    const unsigned qc = ld_relaxed_u32(&S.cs->q_comb);
                    if (qc >= (unsigned)S.n_comb) more = true;
                    else {
                        const int ch = ((((int)qc * S.comb_tok / kRouteBlock) * kFine) / p.nblk) / (kFine / S.K);
                        more = ld_acquire_u32(&S.cs->y_done[ch]) < y_done_target(S, p, ch);
                    }
                }
                g_next = more ? claim() : 0x7fffffff;
            }
        }
        __syncwarp();
    } else if (warp == 0) {
        // ---------------- TMA producer (both CTAs): this CTA's 128 rows of A and its half of B;
        // the warp stays together, one elected thread issues
        bool dead = false;
        uint32_t late_phases = 0u;       // one bit per slot
        while (!dead) {
            bool ok = true;
            if (lane == 0) ok = mbar_wait_cluster(&S.ti_full[ps.slot], ps.slot_phase, p, 35);
            if (!__all_sync(0xffffffffu, ok)) { dead = true; break; }
            const TileInfo ti = S.ti[ps.slot];
            tile_info_landed(ti, &S.scan_w[warp]);
            __syncwarp();
            const uint32_t free_slot = mapa_u32(smem_u32(&S.ti_empty[ps.slot]), 0u);
            uint64_t *const late_bar = &S.ti_late[ps.slot];
            const uint32_t late_bit = 1u << ps.slot;
            const bool late = (ti.chunk & kTileLate) != 0;
            if (lane == 0 && !late) mbar_arrive_remote(free_slot);
            ps.next_slot();
            if (ti.type == 2) break;
            {
                const CUtensorMap *tma_a, *tma_b;
                int arow, brow, arow2 = -1, brow2 = -1;
                // swapped tiles: rows per CTA on the N axis (the MMA's N, a multiple of 16, split in two)
                const bool from_x = S.direct && ti.type == 3;
                const int nhalf = ((((from_x ? p.T : ti.nrows) + 15) >> 4) << 4) >> 1;
                // ... fetched with the smallest box that covers them (the copy engine takes in a fixed number of rows per
                // cycle, so rows nobody reads cost as much as the others), from 65 on with a box of 64 and another one
                const int rest = nhalf > 64 ? nhalf - 64 : nhalf;
                const int bi = rest <= 8 ? 0 : rest <= 16 ? 1 : rest <= 32 ? 2 : 3;
                uint32_t tx = 2u * kStageBytes;                  // bytes landing in both CTAs per k-step
                if (ti.type == 0) {      // leader holds the gate rows of the n-tile, peer the up rows
                    tma_a = &tm->xe; tma_b = &tm->wgu;
                    arow = ti.row0;
                    brow = ti.e * 2 * p.I + ti.n * kTN0 + (int)rank * p.I;
                } else if (ti.type == 1) {   // 256 output columns: leader the first 128 weight rows, peer the rest
                    tma_a = &tm->h; tma_b = &tm->wd;
                    arow = ti.row0;
                    brow = ti.e * p.H + ti.n * 256 + (int)rank * 128;
                } else if (ti.type == 3) {   // M axis: 64 gate rows then 64 up rows of this CTA's 64 h-columns
                    tma_a = &tm->wgu64; tma_b = &tm->xe_n[bi];
                    tx = 2u * (kStageA + (1024u << bi) + (nhalf > 64 ? 8192u : 0u));
                    arow = ti.e * 2 * p.I + ti.n * kTN0 + (int)rank * 64;
                    arow2 = arow + p.I;
                    brow = ti.row0 + (int)rank * nhalf;
                    if (from_x) { tma_b = &tm->x; brow = (int)rank * nhalf; }
                } else {                     // M axis: this CTA's 128 of the n-tile's 256 out-columns
                    tma_a = &tm->wd; tma_b = &tm->h_n[bi];
                    tx = 2u * (kStageA + (1024u << bi) + (nhalf > 64 ? 8192u : 0u));
                    arow = ti.e * p.H + ti.n * 256 + (int)rank * 128;
                    brow = ti.row0 + (int)rank * nhalf;
                }
                const CUtensorMap *tma_b2 = tma_b;      // (swapped tiles of more than 128 rows: rows 64 and up of this half)
                if (ti.type >= 3 && nhalf > 64) {
                    brow2 = brow + 64;
                    tma_b = ti.type == 3 ? &tm->xe_n[3] : &tm->h_n[3];
                }
                // The whole warp walks the loop, one elected thread issues.  The next stage's barrier is looked at
                // before this k-step's copies are issued, so that the answer is there when it is needed (the
                // check took ~140 cycles of every k-step on its own).  Both decisions are made warp-uniform.
                const uint32_t ring = smem_u32(stages), full0 = smem_u32(&S.full[0]), full0_lead = mapa_u32(full0, 0u);
                int kb = 0;
                if (late) {
                    // The weights of the tile's first k-steps, which depend on nothing, go ahead into the ring; its rows follow
                    // into the same stages.  The slot goes back only now, so that its barrier cannot be used twice
                    // before this wait has seen it.
                    const uint32_t lph = (late_phases & late_bit) ? 1u : 0u;
                    const int n = min(ti.nkb, kStages), first = ps.stage;
                    while (kb < n && !__all_sync(0xffffffffu, mbar_test_wait(late_bar, lph))) {
                        if (!__all_sync(0xffffffffu, mbar_wait(&S.empty[ps.stage], ps.stage_phase ^ 1u, p, 33))) { dead = true; break; }
                        if (elect_one()) {
                            const uint32_t sa = ring + (uint32_t)(ps.stage * kStageBytes), lb = full0_lead + (uint32_t)(ps.stage * 8);
                            if (rank == 0) mbar_arrive_expect_tx(&S.full[ps.stage], tx);
                            if (ti.type < 3) tma_load_2d_pair(sa + kStageA, tma_b, kb * kBK, brow, lb);
                            else {
                                tma_load_2d_pair(sa, tma_a, kb * kBK, arow, lb);
                                if (arow2 >= 0) tma_load_2d_pair(sa + kStageA / 2, tma_a, kb * kBK, arow2, lb);
                            }
                        }
                        __syncwarp();
                        ps.next_stage();
                        ++kb;
                    }
                    if (!dead && !__all_sync(0xffffffffu, mbar_wait_cluster(late_bar, lph, p, 36))) dead = true;
                    if (dead) break;
                    late_phases ^= late_bit;
                    if (lane == 0) mbar_arrive_remote(free_slot);
                    for (int i = 0; i < kb; ++i) {
                        const int st = first + i < kStages ? first + i : first + i - kStages;
                        const uint32_t sa = ring + (uint32_t)(st * kStageBytes), lb = full0_lead + (uint32_t)(st * 8);
                        if (elect_one()) {
                            if (ti.type < 3) tma_load_2d_pair(sa, tma_a, i * kBK, arow, lb);
                            else {
                                tma_load_2d_pair(sa + kStageA, tma_b, i * kBK, brow, lb);
                                if (brow2 >= 0) tma_load_2d_pair(sa + kStageA + 8192u, tma_b2, i * kBK, brow2, lb);
                            }
                        }
                        __syncwarp();
                    }
                }
                bool freed = __all_sync(0xffffffffu, mbar_test_wait(&S.empty[ps.stage], ps.stage_phase ^ 1u));
                auto ksteps = [&](auto two_boxes) {
                    for (; kb < ti.nkb; ++kb) {
                        if (!freed && !__all_sync(0xffffffffu, mbar_wait(&S.empty[ps.stage], ps.stage_phase ^ 1u, p, 33))) {
                            dead = true;
                            break;
                        }
                        const uint32_t sa = ring + (uint32_t)(ps.stage * kStageBytes), fo = (uint32_t)(ps.stage * 8);
                        ps.next_stage();
                        freed = __all_sync(0xffffffffu, mbar_test_wait(&S.empty[ps.stage], ps.stage_phase ^ 1u));
                        if (decltype(two_boxes)::value)
                            tma_kstep_pair_b2(sa, tma_a, sa + kStageA, tma_b, kb * kBK, arow, arow2, brow, full0_lead + fo, full0 + fo, tx,
                                              rank == 0 ? 1u : 0u, arow2 >= 0 ? 1u : 0u, tma_b2, brow2);
                        else
                            tma_kstep_pair(sa, tma_a, sa + kStageA, tma_b, kb * kBK, arow, arow2, brow, full0_lead + fo, full0 + fo, tx,
                                           rank == 0 ? 1u : 0u, arow2 >= 0 ? 1u : 0u);
                    }
                };
                if (brow2 >= 0) ksteps(std::true_type()); else ksteps(std::false_type());
            }
        }
        if (dead && lane == 0) linger_after_abort();
        __syncwarp();
    } else if (warp == 1 && rank == 0) {
        // ---------------- MMA issuer (leader only): one elected thread drives both SMs' tensor cores.
        // The whole warp walks the loop so that control flow and operands stay warp-uniform; lane 0
        // does the waiting, the elected lane the issuing.
        bool dead = false;
        const uint64_t desc0 = umma_desc_sw128(smem_u32(stages));      // stage 0, A operand, first 16 of K
        while (!dead) {
            bool ok = true;
            if (lane == 0) ok = mbar_wait(&S.ti_full[ps.slot], ps.slot_phase, p, 40);
            if (!__all_sync(0xffffffffu, ok)) { dead = true; break; }
            const TileInfo ti = S.ti[ps.slot];
            tile_info_landed(ti, &S.scan_w[warp]);
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.ti_empty[ps.slot]);
            ps.next_slot();
            if (ti.type == 2) break;
            // regular tiles: 256 rows x 256 columns; swapped tiles: 256 weight rows x (rows rounded up to 16)
            const int n_op = S.direct && ti.type == 3 ? p.T : ti.nrows;
            const uint32_t idesc = umma_idesc_bf16(2 * kBM, ti.type >= 3 ? (uint32_t)(((n_op + 15) >> 4) << 4) : 256u);
            // timeline record of this tile: extra = time spent waiting for a free accumulator (ns)
            const unsigned long long tm0 = trace_now(p);
            if (lane == 0) ok = mbar_wait_cluster(&S.tmem_empty[ps.acc], ps.acc_phase ^ 1u, p, 41);
            if (!__all_sync(0xffffffffu, ok)) { dead = true; break; }
            tc_fence_after();
            const unsigned long long tm1 = trace_now(p);
            const uint32_t d = S.tmem_base + (uint32_t)ps.acc * 256u;
            bool landed = mbar_test_wait(&S.full[ps.stage], ps.stage_phase);
            for (int kb = 0; kb < ti.nkb; ++kb) {
                // The operands were written by TMA (either CTA's, into its own shared memory) and are
                // read by the tensor cores only: the barrier's completion is all the ordering needed.
                // A wait that gives up has raised the abort flag: the following ones return at once,
                // and the tile's (meaningless) MMAs only touch memory this pair owns.
                // Every lane waits (a lone waiting lane and the re-convergence behind it cost ~75 cycles per
                // k-step), and the next stage's barrier is looked at before this k-step's MMAs are issued.
                if (!landed) ok = mbar_wait(&S.full[ps.stage], ps.stage_phase, p, 42) && ok;
                const uint64_t da = desc0 + (uint64_t)(ps.stage * (kStageBytes >> 4));
                uint64_t *const eb = &S.empty[ps.stage];
                ps.next_stage();
                landed = mbar_test_wait(&S.full[ps.stage], ps.stage_phase);
                tc_mma_kstep_pair(d, da, da + (uint64_t)(kStageA >> 4), idesc, (uint32_t)(kb != 0), eb, 3);
            }
            if (elect_one()) tc_commit_pair(&S.tmem_full[ps.acc], 3);        // accumulators complete in both CTAs
            if (lane == 0)
                trace_ev(p, S, kEvMma, (unsigned)(ti.type << 16 | min(ti.nrows, 65535)), tm0, trace_now(p),
                         (unsigned)min(0xFFFFFFFFull, tm1 - tm0));
            ps.next_acc();
            if (!__all_sync(0xffffffffu, ok)) { dead = true; break; }
        }
        if (dead && lane == 0) linger_after_abort();
        __syncwarp();
    } else if (warp >= 4) {
        // ---------------- epilogue (both CTAs): TMEM -> registers -> (SwiGLU) -> bf16 -> staged store
        const int q = warp & 3;                      // TMEM lane quadrant this warp may read
        bool dead = false;
        uint32_t xg_phase = 0;
        // A release at GPU scope waits until the thread's stores are performed, ~2 us for a tile's
        // worth.  The epilogue warps do not wait: once a tile's stores are issued they tell warp 3,
        // through a shared-memory barrier (which orders their stores before whatever warp 3 does
        // next), which counter the tile arrives on, and go on to the next tile; warp 3 does the
        // release.  Warp q = 0 fills the mailbox, all four warps arrive on it.
        auto post = [&](unsigned *flag, unsigned cnt) -> bool {
            bool ok = true;
            if (lane == 0) {
                if (q == 0) {
                    ok = mbar_wait(&S.rel_empty[ps.rel], ps.rel_phase ^ 1u, p, 56);
                    S.rel_flag[ps.rel] = flag;
                    S.rel_cnt[ps.rel] = cnt;
                }
                mbar_arrive(&S.rel_full[ps.rel]);
            }
            ps.next_rel();
            return !__any_sync(0xffffffffu, !ok);
        };
        while (!dead) {
            if (!mbar_wait_cluster(&S.ti_full[ps.slot], ps.slot_phase, p, 50)) { dead = true; }
            dead = __any_sync(0xffffffffu, dead);
            if (dead) break;
            const TileInfo ti = S.ti[ps.slot];
            tile_info_landed(ti, &S.scan_w[warp]);
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(mapa_u32(smem_u32(&S.ti_empty[ps.slot]), 0u));
            ps.next_slot();
            if (ti.type == 2) { post(nullptr, kRelEnd); break; }
            if (!mbar_wait(&S.tmem_full[ps.acc], ps.acc_phase, p, 51)) { dead = true; }
            dead = __any_sync(0xffffffffu, dead);
            if (dead) break;
            tc_fence_after();
            const unsigned long long te0 = trace_now(p);
            const int rows_valid = ti.nrows - q * 32;          // rows of this warp's quadrant that exist
            const uint32_t epi_stage = smem_u32(stages + kStages * kStageBytes) + (uint32_t)q * 4096u;   // this warp's staging (2 x 2 KB)
            bool acc_released = false;
            auto release_acc = [&]() {       // the tile's last TMEM load has landed: the accumulator goes back to the issuer
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_remote(mapa_u32(smem_u32(&S.tmem_empty[ps.acc]), 0u));
                acc_released = true;
            };
            const uint32_t taddr = S.tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)ps.acc * 256u;
            if (ti.type == 3) {
                // swapped gemm0: lanes 0..63 hold the gate projection of this CTA's 64 h-columns, lanes 64..127 the up
                // projection; TMEM columns are the tile's rows.  Gate warp q and up warp q + 2 trade halves of every 32
                // rows through shared memory, 2 KB each way: the gate warp finishes rows 0..15, the up warp rows
                // 16..31.  (With the gate warps alone doing the arithmetic and the stores 64 rows took 5.5 us; trading 16
                // rows at a time and fetching from tensor memory only when needed, 200 rows took 7.2 us.)  The next 32
                // rows come out of tensor memory meanwhile.  Each warp writes only its own two buffers (its staging
                // area, upper half first), in turn, behind a barrier at which the partner arrived with the buffer's
                // last values in its registers; one more barrier ends the tile.
                //
                // direct: TMEM columns are the batch's tokens (at most 32, so the lower buffers, where the masks are, stay
                // untouched), and the expert's rows are those with a bit in its mask.
                const int up = q >> 1;
                const bool direct = S.direct != 0;
                const uint32_t xmine = smem_u32(stages + kStages * kStageBytes) + (uint32_t)(q * 4096 + lane * 16);
                const uint32_t xtheirs = smem_u32(stages + kStages * kStageBytes) + (uint32_t)((q ^ 2) * 4096 + lane * 16);
                uint64_t *const xbar = &S.xg[q & 1];
                const int ncol = direct ? p.T : ti.nrows;
                unsigned sel = ~0u;                  // direct: the tokens of this expert
                if (direct) {
                    sel = (2u << (p.T - 1)) - 1u;
                    if (ti.e < p.E) sel = *reinterpret_cast<const unsigned *>(stages + kStages * kStageBytes + 8 * ti.e);
                }
                auto meet = [&]() {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(xbar);
                    if (!mbar_wait(xbar, xg_phase, p, 53)) dead = true;
                    dead = __any_sync(0xffffffffu, dead);
                    xg_phase ^= 1u;
                };
                __nv_bfloat16 *dst = p.hbuf + (size_t)ti.row0 * p.I + ti.n * kTN0 + (int)rank * 64 + (q & 1) * 32 + lane;
                uint32_t v[2][32];
                tmem_ld_32x32(taddr, v[0]);
                for (int c0 = 0; c0 < ncol && !dead; c0 += 64) {
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const int c = c0 + 32 * hh;
                        if (c >= ncol || dead) break;
                        tmem_ld_wait32(v[hh]);
                        if (c + 32 < ncol) tmem_ld_32x32(taddr + c + 32, v[hh ^ 1]);
                        else release_acc();
                        const uint32_t xo = hh ? 0u : 2048u;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            if (up) st_shared_v4(xmine + xo + 512u * i, make_uint4(v[hh][4 * i], v[hh][4 * i + 1], v[hh][4 * i + 2], v[hh][4 * i + 3]));
                            else st_shared_v4(xmine + xo + 512u * i, make_uint4(v[hh][16 + 4 * i], v[hh][17 + 4 * i], v[hh][18 + 4 * i], v[hh][19 + 4 * i]));
                        }
                        meet();
                        if (dead) break;
                        // this warp's sixteen rows, as bits (warp-uniform)
                        const int r0 = c + 16 * up;
                        unsigned rows16 = ncol - r0 >= 16 ? 0xFFFFu : (1u << max(0, ncol - r0)) - 1u;
                        int first = r0;
                        if (direct) {
                            rows16 &= sel >> (16 * up);
                            first = up ? __popc(sel & 0xFFFFu) : 0;
                        }
#pragma unroll
                        for (int h8 = 0; h8 < 2; ++h8) {
                            const uint4 t0 = ld_shared_v4(xtheirs + xo + 1024u * h8), t1 = ld_shared_v4(xtheirs + xo + 1024u * h8 + 512u);
                            const uint32_t o[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
                            const unsigned r8 = (rows16 >> (8 * h8)) & 0xFFu;
                            if (r8) {
                                __nv_bfloat16 hv[8];
#pragma unroll
                                for (int i = 0; i < 8; ++i) {
                                    const uint32_t own = up ? v[hh][16 + 8 * h8 + i] : v[hh][8 * h8 + i];
                                    hv[i] = __float2bfloat16_rn(silu_mul(__uint_as_float(up ? o[i] : own), __uint_as_float(up ? own : o[i])));
                                }
                                __nv_bfloat16 *dr = dst + (size_t)(first + __popc(rows16 & (h8 ? 0xFFu : 0u))) * p.I;
#pragma unroll
                                for (int i = 0; i < 8; ++i)
                                    if ((r8 >> i) & 1u) {
                                        *dr = hv[i];
                                        dr += p.I;
                                    }
                            }
                            // (values that no row used have to land all the same before the partner fills the buffer again)
                            *reinterpret_cast<volatile int *>(&S.scan_w[warp]) = (int)(o[0] ^ o[4]);
                        }
                    }
                }
                if (!dead) meet();
                if (dead) break;
            } else if (ti.type == 4) {
                // swapped gemm1: lane = one of this CTA's 128 out-columns, TMEM columns = the tile's rows, 32 at a time with the
                // next 32 on their way while these are converted and stored
                if (ti.n * 256 + (int)rank * 128 < p.H) {
                    __nv_bfloat16 *dst = p.y + (size_t)ti.row0 * p.H + ti.n * 256 + (int)rank * 128 + q * 32 + lane;
                    uint32_t v[2][32];
                    tmem_ld_32x32(taddr, v[0]);
                    for (int c0 = 0; c0 < ti.nrows; c0 += 64) {
#pragma unroll
                        for (int hh = 0; hh < 2; ++hh) {
                            const int c = c0 + 32 * hh;
                            if (c >= ti.nrows) break;
                            tmem_ld_wait32(v[hh]);
                            if (c + 32 < ti.nrows) tmem_ld_32x32(taddr + c + 32, v[hh ^ 1]);
                            else release_acc();
#pragma unroll
                            for (int g = 0; g < 4; ++g) {
                                if (c + 8 * g >= ti.nrows) break;
                                __nv_bfloat16 *dg = dst + (size_t)(c + 8 * g) * p.H;
#pragma unroll
                                for (int j = 0; j < 8; ++j) {
                                    if (c + 8 * g + j < ti.nrows) *dg = __float2bfloat16_rn(__uint_as_float(v[hh][8 * g + j]));
                                    dg += p.H;
                                }
                            }
                        }
                    }
                }
            } else if (rows_valid > 0) {
                // TMEM loads run one (half-)chunk ahead of the conversion and the stores; the
                // accumulator is handed back to the MMA issuer as soon as the last load has landed
                if (ti.type == 0) {
                    // batches of 32 h-columns (32 gate + 32 up accumulator columns), double-buffered:
                    // a TMEM load takes several hundred cycles while the tensor core is busy, so
                    // the next batch is in flight while this one is converted and stored
                    __nv_bfloat16 *dst = p.hbuf + (size_t)(ti.row0 + q * 32) * p.I + (size_t)ti.n * kTN0;
                    uint32_t gr[2][32], ur[2][32], o[16];
                    tmem_ld_32x32(taddr, gr[0]);
                    tmem_ld_32x32(taddr + 128, ur[0]);
#pragma unroll
                    for (int c = 0; c < kTN0 / 32; ++c) {
                        tmem_ld_wait32(gr[c & 1]);
                        reg_fence32(ur[c & 1]);
                        if (c + 1 < kTN0 / 32) {
                            tmem_ld_32x32(taddr + (c + 1) * 32, gr[(c + 1) & 1]);
                            tmem_ld_32x32(taddr + 128 + (c + 1) * 32, ur[(c + 1) & 1]);
                        } else {
                            release_acc();
                        }
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            o[i] = pack_bf16x2(silu_mul(__uint_as_float(gr[c & 1][2 * i]), __uint_as_float(ur[c & 1][2 * i])),
                                               silu_mul(__uint_as_float(gr[c & 1][2 * i + 1]), __uint_as_float(ur[c & 1][2 * i + 1])));
                        staged_store_32(o, epi_stage, dst + c * 32, p.I, rows_valid, lane);
                    }
                } else {
                    // batches of 64 out-columns in two register buffers.  A TMEM load takes most of a
                    // microsecond while the tensor core works on the next tile, and a wait covers every
                    // load in flight, so the tile's epilogue is a chain of load latencies: the batches
                    // are fetched two at a time (two latencies instead of four before the accumulator
                    // can be handed back).
                    __nv_bfloat16 *dst = p.y + (size_t)(ti.row0 + q * 32) * p.H + (size_t)ti.n * 256;
                    const int nb = min(256, p.H - ti.n * 256) / 64;   // the last n-tile may be half wide
                    uint32_t ar[2][64], o[16];
                    tmem_ld_32x64(taddr, ar[0]);
                    if (nb > 1) tmem_ld_32x64(taddr + 64, ar[1]);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (c < nb) {
                            if ((c & 1) == 0) {              // an odd batch lands together with the one before it
                                tmem_ld_wait64(ar[0]);
                                reg_fence64(ar[1]);
                            }
                            if (c + 2 >= nb && !acc_released) release_acc();      // every load of the tile has landed
#pragma unroll
                            for (int hh = 0; hh < 2; ++hh) {
#pragma unroll
                                for (int i = 0; i < 16; ++i)
                                    o[i] = pack_bf16x2(__uint_as_float(ar[c & 1][hh * 32 + 2 * i]),
                                                       __uint_as_float(ar[c & 1][hh * 32 + 2 * i + 1]));
                                staged_store_32(o, epi_stage, dst + c * 64 + hh * 32, p.H, rows_valid, lane);
                            }
                            // this buffer is free again: fetch the batch after next into it
                            if (c + 2 < nb) tmem_ld_32x64(taddr + (c + 2) * 64, ar[c & 1]);
                        }
                    }
                }
            }
            // the accumulator may be overwritten by the next-but-one tile; the rows just stored are read
            // by TMA (gemm1) or by ordinary loads (combine) on other SMs once the counter says so
            const unsigned long long te1 = trace_now(p);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (!acc_released) mbar_arrive_remote(mapa_u32(smem_u32(&S.tmem_empty[ps.acc]), 0u));
                if (q == 0) trace_ev(p, S, kEvGemmEpi, (unsigned)(ti.mb & 0xFFFFFF), te0, trace_now(p),
                                     (unsigned)(ti.type << 16 | (int)min(65535ull, te1 - te0)));
            }
            // every tile makes 4 arrivals from each CTA
            const bool g0 = ti.type == 0 || ti.type == 3;
            if (!post(g0 ? &S.h_ready[ti.rt] : &S.cs->y_done[ti.chunk & (kTileLate - 1)], (unsigned)kEpiWarps)) dead = true;
            ps.next_acc();
        }
    } else if (warp == 3) {
        // ---------------- releasing warp (both CTAs): makes the tiles' arrivals on the ready counters
        int rs = 0;
        uint32_t rph = 0;
        while (true) {
            if (!mbar_wait(&S.rel_full[rs], rph, p, 57)) break;
            unsigned *flag = S.rel_flag[rs];
            const unsigned cnt = S.rel_cnt[rs];
            // both words have landed before the slot goes back (see tile_info_landed)
            *reinterpret_cast<volatile int *>(&S.scan_w[warp]) = (int)cnt ^ (int)(size_t)flag;
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.rel_empty[rs]);
            if (cnt == kRelEnd) break;
            if (lane == 0) {
                fence_proxy_async_global();
                red_release_add_u32(flag, cnt);
            }
            if (++rs == kRel) { rs = 0; rph ^= 1u; }
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();      // nobody targets the other CTA's shared memory or barriers after this
    tc_fence_after();
}

// ------------------------------------------------------------------------------------ the kernel

constexpr int kErrNoPairs = -2;     // reported as "unsupported device"

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
weave_moe_kernel(const __grid_constant__ KParams p, const __grid_constant__ TmaMaps tm)
{
    uint8_t *stages = smem_stages();
    SmemTail &S = smem_tail();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n_sm = (int)gridDim.x;
    const int EE = p.EE;

    // The GEMM phase addresses the neighbouring CTA's shared memory and barriers.  If a launch path
    // ever drops the cluster shape, say so and leave before anything is sent to a peer that is
    // not there (every CTA takes the same branch).
    if (cluster_nctarank() != 2u) {
        if (threadIdx.x == 0) atomicCAS(&p.ctl->status, 0, kErrNoPairs);
        return;
    }

    // The logits of this CTA's first routing block start on their way before anything else: the copy needs
    // no barrier, and the set-up of the barriers and of tensor memory (~1 us) hides part of its latency.
    float *lg_s = reinterpret_cast<float *>(stages + 2048 + kLocalBlocks * kRouteBlock * kMaxTopK * 4);   // [64][route_row_stride(E)]
    {
        const int b_first = p.nblk <= kLocalBlocks ? 0 : (int)blockIdx.x;
        if (b_first < p.nrb) stage_logits_issue(p, b_first, lg_s);
    }

    if (tid == 0) {
        const unsigned odd = (ld_relaxed_u32(&p.ctl->epoch) >> 16) & 1u;
        // (rolled loops: code that runs once per launch runs at the speed of instruction fetch)
#pragma unroll 1
        for (int i = 0; i < kStages; ++i) {
            mbar_init(&S.full[i], 1); mbar_init(&S.empty[i], 1);
            mbar_init(&S.dv_full[i], 1); mbar_init(&S.dv_empty[i], 1);
            mbar_init(&S.cb_full[i], 1); mbar_init(&S.cb_empty[i], kCombWarps);
        }
        // accumulator free: 4 epilogue warps in each CTA of the pair arrive on the leader's barrier
#pragma unroll 1
        for (int i = 0; i < 2; ++i) { mbar_init(&S.tmem_full[i], 1); mbar_init(&S.tmem_empty[i], 2 * kEpiWarps); }
        // tile descriptor consumed: leader's producer + MMA + 4 epilogue warps, peer's producer + 4 warps
#pragma unroll 1
        for (int i = 0; i < kTinfo; ++i) { mbar_init(&S.ti_full[i], 1); mbar_init(&S.ti_late[i], 1); mbar_init(&S.ti_empty[i], 3 + 2 * kEpiWarps); }
        mbar_init(&S.xg[0], 2); mbar_init(&S.xg[1], 2);
#pragma unroll 1
        for (int i = 0; i < kRel; ++i) { mbar_init(&S.rel_full[i], kEpiWarps); mbar_init(&S.rel_empty[i], 1); }
        fence_mbar_init();
        tma_prefetch_desc(&tm.xe); tma_prefetch_desc(&tm.wgu); tma_prefetch_desc(&tm.h); tma_prefetch_desc(&tm.wd);
        tma_prefetch_desc(&tm.wgu64);
        if (p.direct) tma_prefetch_desc(&tm.x);
#pragma unroll 1
        for (int i = 0; i < 4; ++i) { tma_prefetch_desc(&tm.xe_n[i]); tma_prefetch_desc(&tm.h_n[i]); }
        S.cs = reinterpret_cast<CtlSet *>(p.sets + (odd ? ctl_set_bytes(p.nmb_max) : 0));
        S.fcnt = reinterpret_cast<unsigned *>(S.cs + 1);
        S.xe_ready = S.fcnt + kFine * kMaxEE;
        S.h_ready = S.xe_ready + p.nmb_max;
        S.trace_n = 0u;
    }
    if (warp == 1) { tmem_alloc_pair(&S.tmem_base, kTmemCols); tmem_relinquish_pair(); }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();      // the peer's barriers exist before anything is sent to them
    tc_fence_after();
    {
        const size_t bytes = ctl_set_bytes(p.nmb_max);
        uint4 *other = reinterpret_cast<uint4 *>(p.sets + (reinterpret_cast<uint8_t *>(S.cs) == p.sets ? bytes : 0));
        for (size_t i = (size_t)blockIdx.x * kThreads + tid; i < bytes / 16; i += (size_t)n_sm * kThreads)
            other[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    const unsigned long long tk0 = trace_now_t0(p);

    // Routing scratch.  The expert masks of the routing blocks sit in the first half of the epilogue staging
    // area: a small batch's masks are still needed while its dispatch copies run through all the stage
    // buffers.  Everything else lives in the (not yet used) stage buffers.
    unsigned long long *lmask = reinterpret_cast<unsigned long long *>(stages + kStages * kStageBytes);   // [kLocalBlocks][256 + 1 (remote tokens)]
    int *r_base = reinterpret_cast<int *>(stages);                                         // [256]
    int *r_cnt = r_base + kMaxEE;                                                          // [kLocalBlocks][2] local / remote pairs
    int *r_idx = reinterpret_cast<int *>(stages + 2048);                                   // [kLocalBlocks][64][16]; the logits follow (lg_s)
    float *r_p = reinterpret_cast<float *>(stages + 96 * 1024);                            // [64][16] exponentials of the selected logits

    // A batch of at most kLocalBlocks routing blocks is routed by every CTA for itself: no grid barrier and
    // no round trip through global memory stand between the logits and the first dispatch copy.  CTA b
    // writes block b's results down for the combine and the host.  Larger batches: block b is routed by
    // CTA b mod N, the counts meet in global memory behind a grid barrier.
    const bool local_route = p.nblk <= kLocalBlocks;
    const bool ep = p.ep_size > 1;

    // The cost tables do not depend on the routing: this thread's candidate (c, K) asks for its two
    // entries first of all, and (without an expert-parallel share, whose workload descriptors are counted
    // while routing) the plan is chosen where it costs nothing: behind the grid barrier's latency, or, in a
    // batch that has no barrier, while the logits are on their way.
    const int cm_ki = tid & 3, cm_c = p.c_min + (tid >> 2) * p.c_step;
    const bool cm_ok = p.mode == kModeAuto && cm_c >= 2 && cm_c <= p.c_max && cm_c <= n_sm - 2 && (EE << cm_ki) <= kMaxSeg;
    float cm_bw = 0.f, cm_tf = 0.f, cm_bw_n = 0.f, cm_tf_n = 0.f;
    if (cm_ok) { cm_bw = p.bw[cm_c]; cm_tf = p.tf[n_sm - cm_c]; }
    if (p.mode == kModeAuto) { cm_bw_n = p.bw[n_sm]; cm_tf_n = p.tf[n_sm]; }
    unsigned smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    const int die = smid < 1024u ? (int)((p.die_mask[smid >> 5] >> (smid & 31u)) & 1u) : 0;
    const int P = p.T * (p.k + p.S);
    // Eq. 1-3 (single-GPU reading: every pair moves through HBM)
    const float B = (float)(2 * p.H);
    float w_comp = __fmul_rn(__fmul_rn(__fmul_rn((float)P, 6.0f), (float)p.H), (float)p.I);
    float w_disp = __fmul_rn((float)(p.T + P), B);
    float w_comb = __fmul_rn((float)(P + p.T), B);
    ModelArgs ma;
    ma.alpha = p.alpha; ma.eff[0] = p.eff[0]; ma.eff[1] = p.eff[1]; ma.eff[2] = p.eff[2]; ma.eff[3] = p.eff[3];
    ma.kinds = p.kinds; ma.c_min = p.c_min; ma.c_step = p.c_step;
    RouteArgs ra;
    ra.lg_rb = p.lg_rb; ra.T = p.T; ra.E = p.E; ra.k = p.k; ra.ep_size = p.ep_size; ra.ep_rank = p.ep_rank; ra.ep_tshard = p.ep_tshard;
    ra.status = &p.ctl->status; ra.topk_idx = p.topk_idx; ra.gates = p.gates;
    PlanPick pick;
    pick.c = n_sm; pick.ki = 0; pick.kind = kPlanSplit; pick.t = 0.f;
    bool picked = false;

    // ================= phase R: routing
    for (int it = 0;; ++it) {
        const int b = local_route ? it : (int)blockIdx.x + it * n_sm;
        if (b >= p.nrb) break;
        const int slot = local_route ? b : 0;
        unsigned long long *r_mask = lmask + slot * (kMaxEE + 1);
        const bool writer = !local_route || b == (int)blockIdx.x;
        for (int e = tid; e < EE; e += kThreads) r_mask[e] = 0ull;
        if (tid == 0) { r_mask[kMaxEE] = 0ull; r_cnt[2 * slot] = 0; r_cnt[2 * slot + 1] = 0; }
        if (it > 0) stage_logits_issue(p, b, lg_s);      // (the first block's copy was issued at kernel entry)
        if (local_route && !ep && p.mode == kModeAuto) {      // (no barrier to hide it behind: the logits' way in will do)
            pick = model_pick(ma, S, n_sm, w_comp, w_disp, w_comb, cm_ok, cm_bw, cm_tf, cm_bw_n, cm_tf_n);
            picked = true;
        }
        cp_async_wait_all();
        __syncthreads();
        int *idx_b = r_idx + slot * kRouteBlock * kMaxTopK;
        {
            const uint32_t a0 = smem_u32(lg_s), a1 = smem_u32(r_mask), a2 = smem_u32(idx_b), a3 = smem_u32(r_cnt + 2 * slot),
                           a4 = smem_u32(r_p);
            if (ra.lg_rb == 6)
                route_block<true>(6, ra.T, ra.E, ra.k, ra.ep_size, ra.ep_rank, ra.ep_tshard, ra.status, ra.topk_idx, ra.gates, b, a0, a1, a2, a3, a4, writer);
            else
                route_block<false>(ra.lg_rb, ra.T, ra.E, ra.k, ra.ep_size, ra.ep_rank, ra.ep_tshard, ra.status, ra.topk_idx, ra.gates, b, a0, a1, a2, a3, a4, writer);
        }
        __syncthreads();
        if (p.nrb > n_sm) {
            // this CTA routes several blocks and its scratch is reused: the in-block rank of each (token,
            // slot) - tokens before it in the block that chose the same expert - goes out to global memory
            const int tl = tid >> 2, t = b * kRouteBlock + tl;      // (64-token blocks then)
            if (t < p.T)
                for (int j = tid & 3; j < p.k; j += 4) {
                    const int e = idx_b[tl * kMaxTopK + j];     // -1: the expert lives on another rank
                    p.row_of[(size_t)t * p.k + j] = e >= 0 ? __popcll(r_mask[e] & ((1ull << tl) - 1ull)) : -1;
                }
        }
        if (ep && writer && tid == 0) p.uniq_mask[b] = r_mask[kMaxEE];
        if (!local_route) {
            if (ep && tid == 0) {
                const unsigned long long um = r_mask[kMaxEE];
                if (r_cnt[0]) atomicAdd(&S.cs->x_local, (unsigned)r_cnt[0]);
                if (r_cnt[1]) atomicAdd(&S.cs->x_in, (unsigned)r_cnt[1]);
                if (um) atomicAdd(&S.cs->x_in_uniq, (unsigned)__popcll(um));
            }
            const int ntok = min(1 << p.lg_rb, p.T - (b << p.lg_rb));
            const int f = ((b >> (6 - p.lg_rb)) * kFine) / p.nblk;
            for (int e = tid; e < EE; e += kThreads) {
                const int cnt = e < p.E ? __popcll(r_mask[e]) : ntok;
                p.hist[(size_t)b * kMaxEE + e] = cnt;
                if (cnt) atomicAdd(&S.fcnt[f * kMaxEE + e], (unsigned)cnt);
            }
            __syncthreads();      // the scratch is reused by this CTA's next block
        }
    }
    const unsigned long long tk1 = trace_now_t0(p);
    bool alive = true;
    // (arrivals accumulate over the grid barriers of a launch: the later ones count this one in)
    if (!local_route) {
        // the plan is chosen between arriving at the barrier and waiting on it: the arrival's way to L2 and
        // the wait for the slowest routing CTA hide it
        grid_barrier_arrive(S);
        if (!picked && !ep && p.mode == kModeAuto) {
            pick = model_pick(ma, S, n_sm, w_comp, w_disp, w_comb, cm_ok, cm_bw, cm_tf, cm_bw_n, cm_tf_n);
            picked = true;
        }
        alive = grid_barrier_wait(p, S, (unsigned)n_sm, 1);
    }
    const unsigned long long tk2 = trace_now_t0(p);
    if (tid == 0) {
        trace_ev(p, S, kEvRoute, 0u, tk0, tk1, 0u);
        if (!local_route) trace_ev(p, S, kEvBarrier, 1u, tk1, tk2, 0u);
    }

    // ================= set-up: counts, offsets, plan, segment tables (identical on every CTA)
    int cf[kFine];
    int cnt = 0;
    unsigned ep_xl = 0u, ep_xi = 0u, ep_xu = 0u;
    if (local_route) {
#pragma unroll
        for (int f = 0; f < kFine; ++f) cf[f] = 0;
        for (int bb = 0; bb < p.nblk; ++bb) {
            const int fb = (bb * kFine) / p.nblk;
            const int c = tid >= EE ? 0 : tid < p.E ? __popcll(lmask[bb * (kMaxEE + 1) + tid]) : min(kRouteBlock, p.T - bb * kRouteBlock);
#pragma unroll
            for (int f = 0; f < kFine; ++f) if (f == fb) cf[f] += c;
            cnt += c;
            if (ep) {
                ep_xl += (unsigned)r_cnt[2 * bb]; ep_xi += (unsigned)r_cnt[2 * bb + 1];
                ep_xu += (unsigned)__popcll(lmask[bb * (kMaxEE + 1) + kMaxEE]);
            }
        }
    } else {
#pragma unroll
        for (int f = 0; f < kFine; ++f) {
            cf[f] = (alive && tid < EE) ? (int)__ldcg(S.fcnt + f * kMaxEE + tid) : 0;
            cnt += cf[f];
        }
        // (asked for together with the counts: one L2 round trip instead of two)
        if (alive && ep) { ep_xl = __ldcg(&S.cs->x_local); ep_xi = __ldcg(&S.cs->x_in); ep_xu = __ldcg(&S.cs->x_in_uniq); }
    }
    int total_rows;
    const int off = block_excl_scan(cnt, S, total_rows);
    if (tid < EE) S.offsets[tid] = off;
    if (tid == 0) S.offsets[EE] = total_rows;
    if (blockIdx.x == 0 && tid < EE) {
        p.counts[tid] = cnt;
        p.offsets[tid] = off;
        if (tid == 0) p.offsets[EE] = total_rows;
    }
    if (blockIdx.x == 0 && tid == 0) { p.ctl->ep_x_local = ep_xl; p.ctl->ep_x_in = ep_xi; p.ctl->ep_x_in_uniq = ep_xu; }
    int plan_c, plan_ki, plan_steal = 0, plan_kind = kPlanSplit;
    float plan_t = 0.f;
    if (p.mode == kModeAuto) {
        if (ep) {
            // Eq. 1-3 literally: X_local + X_in pairs are computed here, each unique remote token is
            // pulled once, one result goes back per remote pair
            w_comp = __fmul_rn(__fmul_rn(__fmul_rn((float)(ep_xl + ep_xi), 6.0f), (float)p.H), (float)p.I);
            w_disp = __fmul_rn((float)ep_xu, B);
            w_comb = __fmul_rn((float)ep_xi, B);
            pick = model_pick(ma, S, n_sm, w_comp, w_disp, w_comb, cm_ok, cm_bw, cm_tf, cm_bw_n, cm_tf_n);
        }
        plan_c = pick.c; plan_ki = pick.ki; plan_kind = pick.kind; plan_t = pick.t;
        // the steal quota of Eq. 11-14 belongs to the paper's plan kind; in the other kinds the movement
        // SMs have nothing to wait out (they take GEMM tiles while no combine chunk is ready)
        if (plan_kind == kPlanSplit) {
            const float bw_c = __ldg(p.bw + plan_c), tf_c = __ldg(p.tf + n_sm - plan_c);
            // the pair tiles (256 rows) of the layer at the chosen K (a segment = one expert's rows inside
            // one chunk; its last pair tile may be half empty)
            const int Kc = 1 << plan_ki, sh = 3 - plan_ki;
            int acc = 0;
            for (int j = 0; j < Kc; ++j) {
                int rows = 0;
#pragma unroll
                for (int f = 0; f < kFine; ++f) if ((f >> sh) == j) rows += cf[f];
                acc += (rows + 2 * kBM - 1) / (2 * kBM);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) S.red_i[warp][3] = acc;
            __syncthreads();
            int n_tiles = 0;
#pragma unroll
            for (int w = 0; w < kThreads / 32; ++w) n_tiles += S.red_i[w][3];
            n_tiles *= p.nt0 + p.nt1;
            plan_steal = model_n_steal(n_sm, bw_c, tf_c, w_comp, w_disp, w_comb, n_tiles);      // per CTA pair
        }
    } else if (p.mode == kModeFixed) {
        plan_c = max(2, min((p.fixed_c + 1) & ~1, n_sm - 2));     // whole CTA pairs
        plan_ki = p.fixed_K >= 8 ? 3 : p.fixed_K >= 4 ? 2 : p.fixed_K >= 2 ? 1 : 0;
        while (plan_ki > 0 && (EE << plan_ki) > kMaxSeg) --plan_ki;
        plan_steal = max(0, p.fixed_steal);
    } else {
        plan_c = n_sm;
        plan_ki = 0;
        plan_steal = 0;
        plan_kind = kPlanPhased;
    }
    const int K = 1 << plan_ki;
    if (tid == 0) S.elastic = (p.elastic_steal || plan_kind == kPlanRejoin) ? 1 : 0;
    {
        const int sh = 3 - plan_ki;      // fine chunks per chunk = kFine >> plan_ki
        int run_row = tid < EE ? off : 0;
        int mb_base = 0, pt_base = 0;
        for (int j = 0; j < K; ++j) {
            int rows = 0;
#pragma unroll
            for (int f = 0; f < kFine; ++f) if ((f >> sh) == j) rows += cf[f];
            const int mbs = (rows + kBM - 1) / kBM;
            // m-blocks and row tiles of the experts before this one: one packed scan
            unsigned long long tot2;
            const unsigned long long ex2 = block_excl_scan_packed((unsigned long long)mbs | ((unsigned long long)((mbs + 1) >> 1) << 32), S, tot2);
            const int ex = (int)(unsigned)ex2, pex = (int)(ex2 >> 32), tot = (int)(unsigned)tot2, ptot = (int)(tot2 >> 32);
            if (tid < EE) {
                S.seg_mb0[j * EE + tid] = mb_base + ex;
                S.seg_pt0[j * EE + tid] = pt_base + pex;
                S.seg_row0[j * EE + tid] = run_row;
                S.seg_rows[j * EE + tid] = rows;
            }
            // One chunk: the two lists meet at the expert boundary nearest to half of the pair tiles.  Each half of the
            // chip has an L2 of its own that caches what its SMs read, wherever it lives; with whole experts on one
            // half, a weight panel and the expert's rows cross to the other half once instead of being fetched by
            // both (under the power cap every byte moved costs time: Mixtral-shaped T = 4096 2421 -> 2362 us,
            // Qwen3-30B-shaped T = 8192 skewed 778 -> 760; no difference where nothing is shared, T = 64).
            const bool two_lists = K == 1 && ptot >= p.lists_pt;
            if (two_lists && tid < EE) {
                const int mypt = (mbs + 1) >> 1, before = ptot - 2 * pex, after = 2 * (pex + mypt) - ptot;
                if (before >= 0 && after > 0) {
                    S.split_pt = before <= after ? pex : pex + mypt;
                    S.split_seg = before <= after ? tid : tid + 1;
                }
            }
            if (tid == 0) {
                if (!two_lists) { S.split_pt = ptot; S.split_seg = EE; }
                S.chunk_mb0[j] = mb_base;
                S.chunk_pt0[j] = pt_base;
                S.chunk_tile0[j] = pt_base * (p.nt0 + p.nt1);
            }
            run_row += rows;
            mb_base += tot;
            pt_base += ptot;
        }
        if (tid == 0) {
            S.seg_mb0[K * EE] = mb_base;
            S.seg_pt0[K * EE] = pt_base;
            S.chunk_mb0[K] = mb_base;
            S.chunk_pt0[K] = pt_base;
            S.chunk_tile0[K] = pt_base * (p.nt0 + p.nt1);
            S.c = plan_c; S.K = K; S.steal = plan_steal;
            S.nmb = mb_base;
            S.n_gemm = pt_base * (p.nt0 + p.nt1);
            // a small batch is cut into smaller combine tiles (powers of two, so that a tile never
            // straddles two chunks) until every SM has one: its final combine is a latency chain
            // per tile, not a bandwidth problem  (ceil(T / ct) < N  <=>  T <= (N - 1) * ct)
            int ct = kCombTile;
            while (ct > 1 && p.T <= (n_sm - 1) * ct) ct >>= 1;
            if (ct == 1 && p.T > n_sm) ct = 2;      // one round of two tokens each, not two rounds of claims (8 experts, T = 200: 35.1 -> 33.3 us)
            S.comb_tok = ct;
            S.n_comb = (p.T + ct - 1) / ct;
            if (blockIdx.x == 0) {
                p.ctl->plan_c = plan_c; p.ctl->plan_K = K; p.ctl->plan_steal = plan_steal; p.ctl->plan_t = plan_t;
                p.ctl->plan_nmb = mb_base; p.ctl->plan_ngemm = pt_base * (p.nt0 + p.nt1);
                p.ctl->plan_kind = plan_kind;
            }
        }
    }
    __syncthreads();

    const unsigned long long tk3 = trace_now_t0(p);
    if (tid == 0) trace_ev(p, S, kEvSetup, 0u, tk2, tk3, 0u);
    // ================= permutation fix-up: in-block rank + rows of earlier blocks + expert offset
    if (alive) {
        int fixed = 0;
        const bool from_smem = p.nrb <= n_sm;      // this CTA's block is still in its shared memory
        for (int b = blockIdx.x; b < p.nrb; b += n_sm) {
            const int slot = local_route ? b : 0;
            const unsigned long long *r_mask = lmask + slot * (kMaxEE + 1);
            const int *idx_b = r_idx + slot * kRouteBlock * kMaxTopK;
            if (tid < EE) {
                int base = off;
                if (local_route) {
                    for (int bb = 0; bb < b; ++bb) base += __popcll(lmask[bb * (kMaxEE + 1) + tid]);
                } else {
                    const int f = ((b >> (6 - p.lg_rb)) * kFine) / p.nblk;
                    const int bstart = ((f * p.nblk + kFine - 1) / kFine) << (6 - p.lg_rb);
#pragma unroll
                    for (int ff = 0; ff < kFine; ++ff) if (ff < f) base += cf[ff];
#pragma unroll 8
                    for (int bb = bstart; bb < b; ++bb) base += __ldcg(p.hist + (size_t)bb * kMaxEE + tid);
                }
                r_base[tid] = base;
            }
            __syncthreads();
            // the threads that routed a token place its rows (no divisions: this stands between routing and dispatch)
            const int lg = min(5, 8 - p.lg_rb), tl = tid >> lg, t = (b << p.lg_rb) + tl;
            if (t < p.T && tl < (1 << p.lg_rb)) {
                for (int j = tid & ((1 << lg) - 1); j < p.k; j += 1 << lg) {
                    const size_t at = (size_t)t * p.k + j;
                    const int e = from_smem ? idx_b[tl * kMaxTopK + j] : __ldcg(p.topk_idx + at);
                    const int rk = from_smem ? (e >= 0 ? __popcll(r_mask[e] & ((1ull << tl) - 1ull)) : -1) : __ldcg(p.row_of + at);
                    if (rk >= 0) {
                        const int r = rk + r_base[e];
                        p.row_of[at] = r;
                        p.token_of[r] = t;
                    } else if (from_smem) {
                        p.row_of[at] = -1;
                    }
                }
                for (int s = tid & ((1 << lg) - 1); s < p.S; s += 1 << lg) p.token_of[S.offsets[p.E + s] + t] = t;
            }
            __syncthreads();
            ++fixed;
        }
        if (tid == 0 && fixed) red_release_add_u32(&S.cs->fix_done, (unsigned)fixed);
    }

    if (tid == 0) trace_ev(p, S, kEvFixup, 0u, tk3, trace_now(p), 0u);
    // ================= main phases
    bool tmem_held = true;
    if (alive) {
        // The serial schedule is the phased plan with a grid barrier between the phases (one copy of each
        // phase's code serves both).
        const bool serial = p.mode == kModeSerial;
        const unsigned bar0 = p.nblk <= kLocalBlocks ? 0u : (unsigned)n_sm;      // no routing barrier in a small batch
        const bool mover = (int)blockIdx.x < plan_c;      // role from c* and the block index
        // movement CTAs work through the dispatch queue; every GEMM CTA first dispatches one
        // m-block too, so that the first wave of GEMM tiles does not wait for a handful of movers
        // (the mirror image of the final combine on all SMs); the forced "no temporal
        // scheduling" ablation keeps the two groups apart
        // (plan kinds beyond the paper's: every CTA works through the dispatch queue first; in the
        // phased plan every CTA is a "mover" without a steal limit)
        const bool two_roles = plan_kind == kPlanSplit || plan_kind == kPlanRejoin;
        const int dmax = (mover || !two_roles) ? 0x7fffffff : (S.elastic ? 1 : 0);
        const int n_disp = (!two_roles || S.elastic) ? n_sm : plan_c;       // who dispatches at all
        // A batch of at most 32 tokens under the phased plan: N = T columns cost a swapped tile's MMA no more than the
        // expert's few rows do (an instruction takes 48 cycles up to N = 64, and the weights set the pace), so the
        // gate/up tiles multiply ALL tokens, straight from x, and their epilogue keeps the expert's rows.  Nothing waits
        // for the dispatch then (4-5 us).  T = 27 Qwen3-30B-shaped 149.4 -> 146.7 us; of the batches of up to 16 tokens, which
        // gained 6 us, only those of layers too wide for the streaming kernel still come here under AUTO.  At T = 64 a launch by
        // itself gains as much (199.9 -> 197.8) but under load the additional columns and rows cost power (202.8 -> 205.9 after
        // half a second): hence the limit.
        const bool direct = p.direct && plan_kind == kPlanPhased;
        const int budget = (mover && plan_kind != kPlanPhased) ? plan_steal : 0x7fffffff;
        const bool by_token = !two_roles && S.K == 1 && !ep;
        // few tokens per CTA, and every CTA enters the GEMM phase (with elastic stealing off, dispatch-all's movers do not)
        const bool all_gemm = plan_kind == kPlanPhased || S.elastic;
        const bool in_gemm = by_token && all_gemm && p.nrb <= n_sm && (p.lg_rb <= 4 || p.nblk <= kLocalBlocks);
        if (tid == 0) {      // (published by gemm_phase's first barrier)
            S.budget = budget; S.die = die; S.direct = direct ? 1 : 0;
            S.inline_disp = in_gemm && !serial ? (p.nblk <= kLocalBlocks && p.T > kDirectTokens ? 2 : 1) : 0;
        }
        if (by_token) {
            if (!in_gemm) dispatch_tokens(p, S, stages);
            else if (serial && warp >= 8 - kInlineWarps) dispatch_inline(p, S, stages, warp - (8 - kInlineWarps));
        } else if (dmax > 0) {
            dispatch_phase(p, S, stages, dmax, n_disp, p.nblk <= kLocalBlocks);
        }
        if (serial) alive = grid_barrier(p, S, bar0 + (unsigned)n_sm, 2);
        if (alive && (budget > 0 || S.elastic)) {
            gemm_phase(p, S, stages, &tm);
            // (it ends with both CTAs of the pair past their last use of tensor memory and of each other's shared memory)
            if (warp == 1) tmem_dealloc_pair(S.tmem_base, kTmemCols);
            tmem_held = false;
        }
        if (serial) alive = alive && grid_barrier(p, S, bar0 + 2u * (unsigned)n_sm, 3);
        if (alive) combine_phase(p, S, stages);
    }

    // ================= leave
    if (tmem_held) {      // no GEMM phase here: the peer may be in one, and tensor memory is freed by both
        tc_fence_before();
        __syncthreads();
        cluster_sync_all();
        tc_fence_after();
        if (warp == 1) tmem_dealloc_pair(S.tmem_base, kTmemCols);
    }
    if (p.trace) {      // last record of the CTA's slice: how many events were written
        __syncthreads();
        if (tid == 0)
            p.trace[(size_t)blockIdx.x * p.trace_cap + p.trace_cap - 1] =
                make_uint4(min(S.trace_n, (unsigned)p.trace_cap - 1u), 0u, 0u, 0u);
    }
    if (tid == 0) atomicAdd(&p.ctl->epoch, blockIdx.x == 0 ? 65536u - (unsigned)(n_sm - 1) : 1u);
}

// ------------------------------------------------------------------------------------ which half an SM sits on

// One warp per SM: the shortest of kDieTries round trips of an atomic on each of kDieLines lines.  An atomic is done
// in the L2 that the line belongs to: 320-410 cycles from the SMs of that half of the chip, 690-810 from the
// others (148 SMs, idle chip), whereas loads take the same time from both once either side has cached them.
constexpr int kDieLines = 8, kDieTries = 6, kMaxSm = 1024;
__global__ void __launch_bounds__(32, 1) weave_die_probe_kernel(unsigned *lines, int stride_words, unsigned *out)
{
    unsigned smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    if (threadIdx.x != 0 || smid >= (unsigned)kMaxSm) return;
    for (int a = 0; a < kDieLines; ++a) {
        unsigned best = 0xFFFFFFFFu;
        for (int r = 0; r < kDieTries; ++r) {
            const long long t0 = clock64();
            const unsigned v = atomicAdd(lines + a * stride_words, 0u);      // (the lines hold zeros)
            if (v != 0u) out[smid * kDieLines + a] = v;      // never taken: holds the second reading back until the value is here
            const long long t1 = clock64();
            if (r > 0) best = min(best, (unsigned)(t1 - t0));
        }
        out[smid * kDieLines + a] = best;
    }
}

}  // namespace weave
