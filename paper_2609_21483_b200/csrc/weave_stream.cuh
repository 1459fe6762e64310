// A layer of a few tokens: nothing but a stream of weights.
//
// With a handful of rows per expert the general kernel's time is its hand-overs: routing in blocks, tables, tiles that
// are claimed, a cluster's barriers, tiles of 128 and 256 weight rows of which the last round leaves most of the chip
// idle.  Here every CTA routes the whole batch for itself, takes an equal share of the selected experts' weight rows
// and streams it through a ring in shared memory, first gate/up, then down, the latter's weights on their way while the
// former's results are still being exchanged.  Tokens are the N axis of mma.sync.m16n8k16, eight at a time, 16 weight
// rows the M axis; the products are summed 16 of K at a time in ascending order, as the general kernel's
// tcgen05.mma sums them, and the results carry the same bits.
//
// One launch behind another, us, the general kernel / this one, and the time of the bytes: Qwen3-30B-shaped T = 1 37.7 / 25.4 (11.5), T = 8
// 98 / 88.5 (77.8), T = 16 142.9 / 135.3 (117); Qwen3-235B-shaped T = 1 81 / 60 (46.1); Mixtral-shaped T = 1 159 / 119 (107.5), T = 4
// 314 / 295 (269); DSv2-Lite-shaped T = 7 112.5 / 103 (87.1), T = 16 167 / 163; Qwen3.5-35B-shaped T = 12 68.3 / 55.7; 8 experts
// T = 1 25.3 / 14.6, T = 16 27.1 / 20.4.  Bound by HBM but for a chain of 10 us in front of the first weights (launch,
// routing) and around the exchange of h and y.  Measured and left: more than 16 tokens (the rows of x take the ring's
// place; T = 27 163 against 141); a quarter of the units claimed in tiles of one or two (their chain of products is one
// warp's: 282 us where 189 were); a unit per warp with a ring and a claim of its own (every warp holds a unit to the end: 120 / 103).
//
//   warp 0        producer: one tensor copy per ring slot (a tile's rows x 64 or 128 of K)
//   warp 1        makes the finished tiles' arrivals on the ready counters
//   warps 2..7    write down the routing and the dispatched rows
//   warps 8..15   the products: 16 weight rows of the tile each
//   all warps     routing (a warp per token), the final combine
#pragma once
#include <cstddef>

#include "weave_kernel.cuh"

namespace weave {

constexpr int kStThreads = 512;
constexpr int kStTokens = 16;                     // largest batch: two N tiles of a product (see streams())
constexpr int kStMaxSlot = 16384;                 // bytes of a ring slot, at most
constexpr int kStMaxSlots = 16;
constexpr int kStMinRing = 5 * kStMaxSlot, kStGoodRing = 6 * kStMaxSlot, kStWideRing = 8 * kStMaxSlot, kStFullRing = 10 * kStMaxSlot;      // bytes
constexpr int kStArea = kStages * kStageBytes + kEpiStageBytes;      // shared memory in front of the SmemTail: ring, then rows
constexpr int kStUnitG = 8, kStUnitD = 16;        // columns of h / of y that one warp works on: 8 gate + 8 up rows, or 16 rows
constexpr int kStWarps = 8;                       // ... so a tile has up to 8 units
constexpr int kStPad = 16;                        // bytes between two rows of x or h in shared memory (no bank conflicts)
// The rows end over the general kernel's ring barriers: with these 128 bytes eight rows of 7168 columns leave six ring slots
// (DSv3-shaped T = 8: 826 us with five, 783 with six; the general kernel 776).
constexpr int kStRowsEnd = kStArea + 128;
static_assert(offsetof(SmemTail, cs) >= kStRowsEnd - kStArea, "the general kernel's barriers only");

// Boxes of 1 to 8 units: gate_up as [K/64][gate, up][row][64], down as [K/64][row][64], with one or two blocks of K.
constexpr int kStMaps = kStWarps + kStWarps / 2;
struct StreamMaps { CUtensorMap g[kStMaps], d[kStMaps]; };
__host__ __device__ __forceinline__ constexpr int stream_map(int units, int kblocks) { return units - 1 + (kblocks - 1) * kStWarps; }

// This CTA's share of a phase: n units from unit c of active expert a on (the units of all active experts' columns, one
// expert behind the other, are dealt out evenly), in tiles of `cap` units, at most 8.  A tile may go over from one expert to
// the next (w1 units of the first): a tile is a chain of K / 16 dependent products however narrow it is, and two short
// ones where an expert ends cost the CTA 2 to 3 us more than one (T = 1 Qwen3-30B-shaped).
struct StreamShare {
    int a, c, n, cap, upe;      // upe: units per expert
    __device__ __forceinline__ StreamShare() {}
    __device__ __forceinline__ StreamShare(int n_act, int upe_, int cta, int ctas) : upe(upe_)
    {
        const unsigned total = (unsigned)(n_act * upe_);      // (at most 2^18 units, 2^10 CTAs)
        const unsigned u = total * (unsigned)cta / (unsigned)ctas;
        n = (int)(total * (unsigned)(cta + 1) / (unsigned)ctas - u);
        a = (int)(u / (unsigned)upe);
        c = (int)u - a * upe;
        const int tiles = max(1, (n + kStWarps - 1) / kStWarps);
        cap = max(1, (n + tiles - 1) / tiles);
    }
};

struct StreamShared {      // lies over the SmemTail's segment tables, which this kernel does not use
    uint64_t full[kStMaxSlots], empty[kStMaxSlots];
    uint64_t done[2], freed[2];                   // a tile's stores are issued; its arrival is on its way
    unsigned mask[kMaxEE];                        // bit t: token t selected the expert
    int off[kMaxEE + 1];                          // first row of every expert
    int act[kMaxEE];                              // experts with rows
    int n_act, failed;
    unsigned wsum[8];
    int wmax[8];
    StreamShare share[2];                         // gate/up, down
    int idx[kStTokens][kMaxTopK], row[kStTokens][kMaxTopK];
    float gate[kStTokens][kMaxTopK];
    __device__ __forceinline__ int rows(int a) const { return off[act[a] + 1] - off[act[a]]; }
};
constexpr size_t kStSharedAt = (offsetof(SmemTail, seg_mb0) + 1023) / 1024 * 1024;      // (the tail starts on a 1024-byte boundary; on another one,
                                                                                        // the low bits of a barrier's address name it in the wait log)
static_assert(kStSharedAt + sizeof(StreamShared) <= sizeof(SmemTail), "must fit the segment tables");
static_assert(alignof(StreamShared) <= 16, "aligned where it lies");

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void *map, int c0, int c1, int c2, int c3, uint64_t *bar)
{
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2,%3,%4,%5}], [%6];"
                 ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const void *map, int c0, int c1, int c2, uint64_t *bar)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2,%3,%4}], [%5];"
                 ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar)) : "memory");
}

struct StreamWalk : StreamShare {
    int w, w1, at_a, at_c;      // the current tile: units, units of its first expert, that expert and the first unit of it
    __device__ __forceinline__ StreamWalk(const StreamShare &s) : StreamShare(s) {}
    // rows: rows of h that fit shared memory (0: no limit)
    __device__ __forceinline__ bool next(const StreamShared &X, int rows)
    {
        if (n == 0) return false;
        at_a = a;
        at_c = c;
        w = min(cap, n);
        w1 = min(w, upe - c);
        if (rows && w1 < w && X.rows(a) + X.rows(a + 1) > rows) w = w1;
        n -= w;
        c += w;
        if (c >= upe) { c -= upe; ++a; }
        return true;
    }
};

// Top-k of one token by a warp: lane l holds experts l, l + 32, ... as order keys in registers; order, ties and gates as
// in route_block.
__device__ __forceinline__ void stream_route(const KParams &p, StreamShared &X, int t, const float (&lg)[8])
{
    const int lane = threadIdx.x & 31;
    unsigned key[8], bk = 0u;
    int bi;
    bool bad = false;
    auto best = [&]() {      // the lane's largest key; of equal ones the first
        bk = 0u;
#pragma unroll
        for (int i = 0; i < 8; ++i) bk = max(bk, key[i]);
        bi = 7;
#pragma unroll
        for (int i = 6; i >= 0; --i) bi = key[i] == bk ? i : bi;
    };
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int e = lane + 32 * i;
        float x = lg[i];
        const bool nf = !(fabsf(x) <= 3.402823466e38f);
        bad = bad || (e < p.E && nf);
        x = nf ? -3.402823466e38f : x;
        key[i] = e < p.E ? float_order_key(__fadd_rn(x, 0.0f)) : 0u;
    }
    best();
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicCAS(&p.ctl->status, 0, kErrNonFinite);
    float mine = 0.f;      // lane j: logit and expert of slot j
    int my_e = 0;
#pragma unroll 1
    for (int j = 0; j < p.k; ++j) {
        const unsigned top = __reduce_max_sync(0xffffffffu, bk), eq = __ballot_sync(0xffffffffu, bk == top);
        int win = __ffs((int)eq) - 1;
        if (eq & (eq - 1u)) win = (int)(__reduce_min_sync(0xffffffffu, bk == top ? (unsigned)(lane + 32 * bi) : 0x7fffffffu) & 31u);
        const int hi = win + 32 * __shfl_sync(0xffffffffu, bi, win);
        if (lane == j) { mine = float_from_order_key(top); my_e = hi; }
#pragma unroll
        for (int i = 0; i < 8; ++i) key[i] = lane == win && bi == i ? 0u : key[i];
        best();
    }
    mine = expf(mine - __shfl_sync(0xffffffffu, mine, 0));
    float sum = 0.f;
#pragma unroll 1
    for (int j = 0; j < p.k; ++j) sum += __shfl_sync(0xffffffffu, mine, j);      // slot order
    if (lane < p.k) {
        atomicOr(&X.mask[my_e], 1u << t);
        X.idx[t][lane] = my_e;
        X.gate[t][lane] = __fdiv_rn(mine, sum);
    }
}

// One tile for a warp: 16 weight rows x 8 tokens, KB blocks of 64 of K per ring slot.  a_off: this lane's ldmatrix row in a slot,
// blk: bytes of a block of K in the slot, b_row: this lane's row of x or h.  A block's operands are fetched between the
// products of the block before: the chain of dependent products (and nothing else) sets the pace.
// False: a wait has failed, and the results are not to be used.  (The rest of the tile is run through; slots are handed back all the
// same, to a producer that is on its way out.)
struct StreamRing { uint32_t base, bytes; int slots, slot; uint32_t ph; };
template <int KB>
__device__ __forceinline__ bool stream_tile(const KParams &p, StreamShared &X, StreamRing &r, int K, bool works, uint32_t a_off, uint32_t blk,
                                            uint32_t b_row, float (&acc)[4])
{
    const int lane = threadIdx.x & 31;
    const uint32_t sw = (uint32_t)(lane & 7), kh = (uint32_t)(lane >> 4);
    bool ok = true;
    uint32_t a[2][4][4], b[2][2][4], a0 = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = 0.f;
    auto arrived = [&](int j) {      // block j (of parity j & 1): its slot is there
        if (KB == 1 || (j & 1) == 0) {
            ok = mbar_wait(&X.full[r.slot], r.ph, p, 61) && ok;
            a0 = r.base + (uint32_t)r.slot * r.bytes + a_off;
            if (++r.slot == r.slots) { r.slot = 0; r.ph ^= 1u; }
        } else a0 += blk;
    };
    auto fetch = [&](int buf, int j, int s) {      // 16 of K
        ldmatrix_x4(a0 + (((2u * (uint32_t)s + kh) ^ sw) << 4), a[buf][s]);
        if ((s & 1) == 0) ldmatrix_x4(b_row + (uint32_t)(j * 128 + s * 32), b[buf][s >> 1]);
    };
    auto free_slot = [&](int slot) {      // the slot's values are in registers
        __syncwarp();
        if (lane == 0) mbar_arrive(&X.empty[slot]);
    };
    const int nb = K / 64;      // even
    int held = r.slot;
    arrived(0);
#pragma unroll
    for (int s = 0; s < 4; ++s) fetch(0, 0, s);
    for (int j = 0; j < nb; j += 2) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const bool more = h == 0 || j + 2 < nb;
            const int last = held;
            if (more) {
                if (KB == 1 || h == 1) held = r.slot;
                arrived(j + h + 1);
            }
            if (works) {
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    mma_16816(acc, a[h][s], b[h][s >> 1][2 * (s & 1)], b[h][s >> 1][2 * (s & 1) + 1]);
                    if (more) fetch(h ^ 1, j + h + 1, s);
                }
            }
            if (KB == 1 || h == 1) free_slot(last);
        }
    }
    return ok;
}

// The same for an expert of 9 to 16 rows, without the look ahead (registers).
template <int KB>
__device__ __forceinline__ bool stream_tile_16(const KParams &p, StreamShared &X, StreamRing &r, int K, bool works, uint32_t a_off, uint32_t blk,
                                               uint32_t b_row, uint32_t b_row2, float (&acc)[4], float (&acc2)[4])
{
    const int lane = threadIdx.x & 31;
    const uint32_t sw = (uint32_t)(lane & 7), kh = (uint32_t)(lane >> 4);
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = acc2[i] = 0.f;
#pragma unroll 1
    for (int j = 0; j < K / 64; j += KB) {
        ok = mbar_wait(&X.full[r.slot], r.ph, p, 61) && ok;
        if (works) {
#pragma unroll
            for (int kb = 0; kb < KB; ++kb) {
                const uint32_t a0 = r.base + (uint32_t)r.slot * r.bytes + a_off + (uint32_t)kb * blk;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t a[2][4], b[4], b2[4];
                    ldmatrix_x4(b_row + (uint32_t)((j + kb) * 128 + h * 64), b);
                    ldmatrix_x4(b_row2 + (uint32_t)((j + kb) * 128 + h * 64), b2);
#pragma unroll
                    for (int s = 0; s < 2; ++s) ldmatrix_x4(a0 + (((2u * (uint32_t)(2 * h + s) + kh) ^ sw) << 4), a[s]);
#pragma unroll
                    for (int s = 0; s < 2; ++s) {
                        mma_16816(acc, a[s], b[2 * s], b[2 * s + 1]);
                        mma_16816(acc2, a[s], b2[2 * s], b2[2 * s + 1]);
                    }
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&X.empty[r.slot]);
        if (++r.slot == r.slots) { r.slot = 0; r.ph ^= 1u; }
    }
    return ok;
}

// kWide: 9 to 16 tokens (a kernel of its own: with the second N tile in it the smaller batches take 1 to 2 % longer);
// kTrace: with the timeline's records (apart, so that the kernels that are timed carry none of it)
template <bool kWide, bool kTrace>
__global__ void __launch_bounds__(kStThreads, 1)
weave_stream_kernel(const __grid_constant__ KParams p, const __grid_constant__ StreamMaps tm)
{
    uint8_t *stages = smem_stages();
    SmemTail &S = smem_tail();
    StreamShared &X = *reinterpret_cast<StreamShared *>(reinterpret_cast<uint8_t *>(&S) + kStSharedAt);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cta = (int)blockIdx.x, ctas = (int)gridDim.x;
    const uint32_t ring = smem_u32(stages), area_end = ring + (uint32_t)kStRowsEnd;

    auto now = [] { return kTrace ? globaltimer_ns() : 0ull; };
    const unsigned long long tk0 = now();
    // the logits of this warp's token and the batch's rows of x start on their way before anything else
    float lg[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int e = lane + 32 * i;
        lg[i] = warp < p.T && e < p.E ? __ldcg(p.logits + (size_t)warp * p.E + e) : 0.f;
    }
    const uint32_t pitch_x = (uint32_t)p.H * 2u + kStPad, pitch_h = (uint32_t)p.I * 2u + kStPad, x_s = area_end - (uint32_t)p.T * pitch_x;
    if (warp > 0) {
        const int per_row = p.H >> 3;
        for (int t = 0; t < p.T; ++t)
            for (int c = tid - 32; c < per_row; c += kStThreads - 32)
                cp_async_16(x_s + (uint32_t)t * pitch_x + (uint32_t)(c * 16), p.x + (size_t)t * p.H + c * 8);
    }
    if (tid == 0) {
        const unsigned odd = (ld_relaxed_u32(&p.ctl->epoch) >> 16) & 1u;
        S.cs = reinterpret_cast<CtlSet *>(p.sets + (odd ? ctl_set_bytes(p.nmb_max) : 0));
        S.h_ready = reinterpret_cast<unsigned *>(S.cs + 1) + kFine * kMaxEE + p.nmb_max;
        X.failed = 0;
        if (kTrace) S.trace_n = 0;
    }
    if (warp == 14 && lane < kStMaxSlots) { mbar_init(&X.full[lane], 1); mbar_init(&X.empty[lane], kStWarps); }
    if (warp == 14 && lane >= 30) { mbar_init(&X.done[lane - 30], kStWarps); mbar_init(&X.freed[lane - 30], 1); }
    if (warp == 14) fence_mbar_init();
    if (warp == 15 && lane < 2 * kStMaps) tma_prefetch_desc(lane < kStMaps ? &tm.g[lane] : &tm.d[lane - kStMaps]);
    if (tid < kMaxEE) X.mask[tid] = tid >= p.E && tid < p.EE ? (2u << (p.T - 1)) - 1u : 0u;
    __syncthreads();
    {
        const size_t bytes = ctl_set_bytes(p.nmb_max);
        uint4 *other = reinterpret_cast<uint4 *>(p.sets + (reinterpret_cast<uint8_t *>(S.cs) == p.sets ? bytes : 0));
        for (size_t i = (size_t)cta * kStThreads + tid; i < bytes / 16; i += (size_t)ctas * kStThreads)
            other[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    // ================= routing, counts, offsets, active experts
    if (warp < p.T) stream_route(p, X, warp, lg);
    __syncthreads();
    const unsigned long long tk1 = now();
    unsigned v = 0, inc = 0;      // rows | (has rows) << 16
    if (warp < kMaxEE / 32) {
        const unsigned n = (unsigned)__popc(X.mask[tid]);
        v = n | (n ? 0x10000u : 0u);
        inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned q = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += q;
        }
        if (lane == 31) X.wsum[warp] = inc;
        const int most = (int)__reduce_max_sync(0xffffffffu, n);
        if (lane == 0) X.wmax[warp] = most;
    }
    __syncthreads();
    if (warp < kMaxEE / 32) {
        unsigned base = inc - v;
#pragma unroll
        for (int w = 0; w < kMaxEE / 32; ++w) base += w < warp ? X.wsum[w] : 0u;
        X.off[tid] = (int)(base & 0xFFFFu);
        if (v) X.act[base >> 16] = tid;
        if (tid == kMaxEE - 1) { X.off[kMaxEE] = (int)((base + v) & 0xFFFFu); X.n_act = (int)((base + v) >> 16); }
        if (cta == 0) {
            if (tid < p.EE) { p.counts[tid] = (int)(v & 0xFFFFu); p.offsets[tid] = (int)(base & 0xFFFFu); }
            if (tid == p.EE - 1) p.offsets[p.EE] = (int)((base + v) & 0xFFFFu);
        }
    }
    __syncthreads();
    const int A = X.n_act;
    if (lane == 0 && (warp == 0 || warp == 8)) X.share[warp >> 3] = StreamShare(A, warp ? p.H / kStUnitD : p.I / kStUnitG, cta, ctas);
    __syncthreads();
    // Shared memory: the ring, then the rows of x and, later, in the same place, of h: of one expert, of two where the ring stays
    // deep all the same (fewer than about 160 KB on their way make the stream slower).
    int most = 0;      // rows of an expert
#pragma unroll
    for (int w = 0; w < kMaxEE / 32; ++w) most = max(most, X.wmax[w]);
    int rows_h = 2 * most;
    if (kStRowsEnd - rows_h * (int)pitch_h < kStFullRing) rows_h = most;
    const int ring_bytes = (kStRowsEnd - max(p.T * (int)pitch_x, rows_h * (int)pitch_h)) & ~2047;
    const uint32_t h_s = ring + (uint32_t)ring_bytes;
    // The ring's slots, as large as this CTA's widest tiles want them: a block of K of five units and more, two of fewer.  (With
    // slots for eight units throughout, a share of ten in two tiles of five had 120 KB of the ring's 192 in flight.)
    const int cap0 = X.share[0].cap, cap1 = X.share[1].cap;
    const int slot_units = max(cap0 <= kStWarps / 2 ? 2 * cap0 : cap0, cap1 <= kStWarps / 2 ? 2 * cap1 : cap1);
    const int slots = min(kStMaxSlots, ring_bytes / (slot_units * 2048));
    if (kTrace && tid == 0) {
        trace_ev(p, S, kEvRoute, 0u, tk0, tk1, 0u);
        trace_ev(p, S, kEvSetup, 0u, tk1, now(), 0u);
    }

    if (warp == 0) {
        // ---------------- producer
        if (lane == 0) {
            int slot = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int phase = 0; phase < 2 && ok; ++phase) {
                StreamWalk wk(X.share[phase]);
                while (ok && wk.next(X, phase ? rows_h : 0)) {
                    const int kb = 2 * wk.w <= slot_units ? 2 : 1, nk = (phase ? p.I : p.H) / (64 * kb), w2 = wk.w - wk.w1;
                    const int e1 = X.act[wk.at_a], e2 = w2 ? X.act[wk.at_a + 1] : 0;
                    const int row1 = phase ? e1 * p.H + wk.at_c * kStUnitD : e1 * 2 * p.I + wk.at_c * kStUnitG, row2 = phase ? e2 * p.H : e2 * 2 * p.I;
                    const CUtensorMap *maps = phase ? tm.d : tm.g;
                    const CUtensorMap *map1 = maps + stream_map(wk.w1, kb), *map2 = w2 ? maps + stream_map(w2, kb) : nullptr;
                    for (int kk = 0; kk < nk; ++kk) {
                        if (!mbar_wait(&X.empty[slot], ph ^ 1u, p, 60)) { ok = false; break; }
                        mbar_arrive_expect_tx(&X.full[slot], (uint32_t)(wk.w * kb * 2048));
                        const uint32_t dst = ring + (uint32_t)(slot * slot_units * 2048), dst2 = dst + (uint32_t)(wk.w1 * kb * 2048);
                        if (phase) {
                            tma_load_3d(dst, map1, 0, row1, kb * kk, &X.full[slot]);
                            if (w2) tma_load_3d(dst2, map2, 0, row2, kb * kk, &X.full[slot]);
                        } else {
                            tma_load_4d(dst, map1, 0, row1, 0, kb * kk, &X.full[slot]);
                            if (w2) tma_load_4d(dst2, map2, 0, row2, 0, kb * kk, &X.full[slot]);
                        }
                        if (++slot == slots) { slot = 0; ph ^= 1u; }
                    }
                }
            }
            if (!ok) X.failed = 1;
        }
        __syncwarp();
    } else {
        cp_async_wait_all();
        named_barrier_sync<1, kStThreads - 32>();      // x is in shared memory
        if (warp == 1) {
            // ---------------- a release at GPU scope waits until the tile's stores are performed: not the products' business (made by
            // their own warps: T = 8 Qwen3-30B-shaped 87.5 -> 95.3 us)
            if (lane == 0) {
                int tile = 0;
                bool ok = true;
                for (int phase = 0; phase < 2 && ok; ++phase) {
                    StreamWalk wk(X.share[phase]);
                    for (; ok && wk.next(X, phase ? rows_h : 0); ++tile) {
                        ok = mbar_wait(&X.done[tile & 1], (uint32_t)((tile >> 1) & 1), p, 64);
                        if (!ok) break;
                        // (the test hook's m-block is an active expert here)
                        if (phase || wk.at_a != p.withhold_mb) red_release_add_u32(phase ? &S.cs->y_done[0] : &S.h_ready[wk.at_a], (unsigned)(phase ? wk.w : wk.w1));
                        if (!phase && wk.w1 < wk.w && wk.at_a + 1 != p.withhold_mb) red_release_add_u32(&S.h_ready[wk.at_a + 1], (unsigned)(wk.w - wk.w1));
                        mbar_arrive(&X.freed[tile & 1]);
                    }
                }
                if (!ok) X.failed = 1;
            }
            __syncwarp();
        } else if (warp < 8) {
            // ---------------- rows of the tokens' slots; what other kernels and the host may read
            for (int t = warp - 2; t < p.T; t += 6) {
                if (lane < p.k) {
                    const int e = X.idx[t][lane], row = X.off[e] + __popc(X.mask[e] & ((1u << t) - 1u));
                    X.row[t][lane] = row;
                    if (cta == t % ctas) {
                        p.topk_idx[t * p.k + lane] = e;
                        p.gates[t * p.k + lane] = X.gate[t][lane];
                        p.row_of[t * p.k + lane] = row;
                        p.token_of[row] = t;
                    }
                } else if (lane < p.k + p.S && cta == t % ctas) p.token_of[X.off[p.E + lane - p.k] + t] = t;
            }
            if (cta == ctas - 1 && tid == 64) {
                p.ctl->plan_c = ctas; p.ctl->plan_K = 1; p.ctl->plan_steal = 0; p.ctl->plan_t = p.st_plan_t; p.ctl->plan_kind = kPlanPhased;
                p.ctl->ep_x_local = 0u; p.ctl->ep_x_in = 0u; p.ctl->ep_x_in_uniq = 0u;
                p.ctl->plan_nmb = A;      // (at most 16 rows per expert: one m-block and one row tile each)
                p.ctl->plan_ngemm = A * (p.nt0 + p.nt1);
            }
            // the dispatched rows, row r by CTA r mod N
            const int P = p.T * (p.k + p.S);
            for (int r = cta + ctas * (warp - 2); r < P; r += ctas * 6) {
                const unsigned long long td = now();
                int lo = 0, hi = p.EE;      // largest expert that starts at or before r (empty ones share a start with the next)
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (X.off[mid] <= r) lo = mid; else hi = mid;
                }
                const int t = (int)__fns(X.mask[lo], 0u, r - X.off[lo] + 1);
                const uint4 *src = reinterpret_cast<const uint4 *>(p.x + (size_t)t * p.H);
                uint4 *dst = reinterpret_cast<uint4 *>(p.xe + (size_t)r * p.H);
                for (int c = lane; c < (p.H >> 3); c += 32) dst[c] = __ldcg(src + c);      // (x may be the output: not read-only)
                if (kTrace && lane == 0) trace_ev(p, S, kEvDispatch, (unsigned)r, td, now(), 0u);
            }
            // (counted in with y: nothing is written to `out`, which may be x itself, before its last reader is done)
            __syncwarp();
            if (lane == 0) red_release_add_u32(&S.cs->y_done[0], 1u);
        } else {
            // ---------------- the products.  Once a wait of a warp has failed (`ok`: the warp's at the start of a tile) it stores and
            // hands over nothing; it goes through the tiles that are left as ones of no length, to meet the others at the barriers
            // around a reload of h.  (A jump over them costs 8 experts, T = 2 15.2 -> 15.9 us; the wide kernel 1 to 1.5 %.)
            const int wi = warp - 8;
            int tile = 0;
            StreamRing r = {ring, (uint32_t)(slot_units * 2048), slots, 0, 0u};
            bool ok = true;
            for (int phase = 0; phase < 2; ++phase) {
                StreamWalk wk(X.share[phase]);
                const uint32_t pitch = phase ? pitch_h : pitch_x, rows_s = phase ? h_s : x_s;
                int first = -1, second = -1;      // active experts whose rows of h are in shared memory, one behind the other
                for (; wk.next(X, phase ? rows_h : 0); ++tile) {
                    const bool two = wk.w1 < wk.w;
                    const unsigned long long th = now();
                    const int kb = 2 * wk.w <= slot_units ? 2 : 1;
                    if (phase && ((wk.at_a != first && wk.at_a != second) || (two && wk.at_a + 1 != second))) {
                        // the next rows of h, once all of them are there and nobody reads what they replace
                        first = wk.at_a; second = two ? wk.at_a + 1 : -1;
                        named_barrier_sync<2, kStWarps * 32>();
                        if (lane == 0 && ok) ok = flag_wait_ge(&S.h_ready[first], (unsigned)(p.I / kStUnitG), p, 62);
                        if (lane == 0 && ok && two) ok = flag_wait_ge(&S.h_ready[second], (unsigned)(p.I / kStUnitG), p, 62);
                        ok = __all_sync(0xffffffffu, ok);
                        const int per_row = p.I >> 3, ctid = tid - 256, n = X.rows(first) + (two ? X.rows(second) : 0);
                        const __nv_bfloat16 *src = p.hbuf + (size_t)X.off[X.act[first]] * p.I;      // (the two experts' rows are neighbours)
                        for (int t = 0; t < n && ok; ++t)
                            for (int c = ctid; c < per_row; c += kStWarps * 32)
                                cp_async_16(rows_s + (uint32_t)t * pitch + (uint32_t)(c * 16), src + (size_t)t * p.I + c * 8);
                        cp_async_wait_all();
                        named_barrier_sync<2, kStWarps * 32>();
                    }
                    const unsigned long long tt = now();
                    // this warp's unit: unit li of the ones that the tile has of active expert a
                    const bool works = wi < wk.w, later = works && wi >= wk.w1;
                    const int a = later ? wk.at_a + 1 : wk.at_a, li = later ? wi - wk.w1 : wi, wp = later ? wk.w - wk.w1 : wk.w1;
                    const int unit = later ? li : wk.at_c + li, e = X.act[a], n_e = X.rows(a), row0 = X.off[e];
                    const int i8 = lane & 7;
                    const int src_row = phase ? (a == second ? X.rows(first) : 0) + (i8 < n_e ? i8 : 0) : (int)__fns(X.mask[e], 0u, i8 < n_e ? i8 + 1 : 1);
                    const uint32_t b_row = rows_s + (uint32_t)src_row * pitch + (uint32_t)((lane >> 3) * 16);
                    const uint32_t half = (uint32_t)((lane >> 3) & 1);      // rows 8..15 of the warp's sixteen
                    const uint32_t part = later ? (uint32_t)(wk.w1 * kb * 2048) : 0u;
                    const uint32_t a_off = part + (phase ? (uint32_t)(li * 16 + i8 + 8 * (int)half) * 128u : (uint32_t)(li * 8 + i8) * 128u + half * (uint32_t)(wp * 1024));
                    const uint32_t blk = (uint32_t)(wp * 2048);
                    const int K = ok ? (phase ? p.I : p.H) : 0;
                    float acc[kWide ? 2 : 1][4];
                    if (!kWide || n_e <= 8)
                        ok = (kb == 2 ? stream_tile<2>(p, X, r, K, works, a_off, blk, b_row, acc[0]) : stream_tile<1>(p, X, r, K, works, a_off, blk, b_row, acc[0])) && ok;
                    else {
                        const int i16 = i8 + 8 < n_e ? i8 + 8 : 0;
                        const int src_row2 = phase ? (a == second ? X.rows(first) : 0) + i16 : (int)__fns(X.mask[e], 0u, i16 + 1);
                        const uint32_t b_row2 = rows_s + (uint32_t)src_row2 * pitch + (uint32_t)((lane >> 3) * 16);
                        ok = (kb == 2 ? stream_tile_16<2>(p, X, r, K, works, a_off, blk, b_row, b_row2, acc[0], acc[kWide])
                                      : stream_tile_16<1>(p, X, r, K, works, a_off, blk, b_row, b_row2, acc[0], acc[kWide])) && ok;
                    }
                    if (lane == 0 && ok && tile >= 2) ok = mbar_wait(&X.freed[tile & 1], (uint32_t)(((tile >> 1) - 1) & 1), p, 65);
                    ok = __all_sync(0xffffffffu, ok);
                    if (works && ok) {
                        const int col = (phase ? unit * kStUnitD : unit * kStUnitG) + (lane >> 2);
#pragma unroll
                        for (int i = 0; i < (kWide ? 4 : 2); ++i) {      // this lane has rows 2q and 2q + 1 of every eight of the expert
                            const int t = 2 * (lane & 3) + (i & 1) + 8 * (i >> 1);
                            if (t < n_e) {
                                if (phase) {
                                    __nv_bfloat16 *d = p.y + (size_t)(row0 + t) * p.H + col;
                                    d[0] = __float2bfloat16_rn(acc[i >> 1][i & 1]);
                                    d[8] = __float2bfloat16_rn(acc[i >> 1][2 + (i & 1)]);
                                } else p.hbuf[(size_t)(row0 + t) * p.I + col] = __float2bfloat16_rn(silu_mul(acc[i >> 1][i & 1], acc[i >> 1][2 + (i & 1)]));
                            }
                        }
                    }
                    __syncwarp();
                    if (lane == 0 && ok) mbar_arrive(&X.done[tile & 1]);
                    if (kTrace && lane == 0 && ok && wi == 0) trace_ev(p, S, kEvStream, (unsigned)(phase << 16 | wk.w), tt, now(), (unsigned)(tt - th));
                }
            }
            if (!ok) X.failed = 1;
        }
    }

    // ================= combine: out[t] = sum over the slots, in slot order, then the shared experts
    __syncthreads();
    const unsigned long long tw = now();
    if (tid == 0 && !flag_wait_ge(&S.cs->y_done[0], (unsigned)(A * (p.H / kStUnitD) + 6 * ctas), p, 63)) X.failed = 1;
    __syncthreads();
    const unsigned long long tc = now();
    if (!X.failed) {
        const int vecs = p.H >> 3, total = p.T * vecs;      // 16-byte pieces, four neighbours to a CTA
        for (int i = ((tid >> 2) * ctas + cta) * 4 + (tid & 3); i < total; i += kStThreads * ctas) {
            const int t = i / vecs, c = i - t * vecs;
            float a0[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) a0[q] = 0.f;
#pragma unroll 4
            for (int j = 0; j < p.k + p.S; ++j) {
                const int row = j < p.k ? X.row[t][j] : X.off[p.E + j - p.k] + t;
                const float gw = j < p.k ? X.gate[t][j] : 1.0f;
                const uint4 q4 = __ldcg(reinterpret_cast<const uint4 *>(p.y + (size_t)row * p.H) + c);
                a0[0] = fmaf(gw, bf16lo_to_f32(q4.x), a0[0]); a0[1] = fmaf(gw, bf16hi_to_f32(q4.x), a0[1]);
                a0[2] = fmaf(gw, bf16lo_to_f32(q4.y), a0[2]); a0[3] = fmaf(gw, bf16hi_to_f32(q4.y), a0[3]);
                a0[4] = fmaf(gw, bf16lo_to_f32(q4.z), a0[4]); a0[5] = fmaf(gw, bf16hi_to_f32(q4.z), a0[5]);
                a0[6] = fmaf(gw, bf16lo_to_f32(q4.w), a0[6]); a0[7] = fmaf(gw, bf16hi_to_f32(q4.w), a0[7]);
            }
            st_cs_v4(p.out + (size_t)t * p.H + c * 8, make_uint4(pack_bf16x2(a0[0], a0[1]), pack_bf16x2(a0[2], a0[3]),
                                                                 pack_bf16x2(a0[4], a0[5]), pack_bf16x2(a0[6], a0[7])));
        }
    } else if (tid == 0) linger_after_abort();      // copies may still be landing in this CTA's shared memory
    if (kTrace) {      // the slice's last record: how many there are
        __syncthreads();
        if (tid == 0) {
            trace_ev(p, S, kEvWaitChunk, 0u, tw, tc, 0u);
            trace_ev(p, S, kEvCombine, (unsigned)cta, tc, now(), 0u);
            p.trace[(size_t)cta * p.trace_cap + p.trace_cap - 1] = make_uint4(min(S.trace_n, (unsigned)p.trace_cap - 1u), 0u, 0u, 0u);
        }
    }
    if (tid == 0) atomicAdd(&p.ctl->epoch, cta == 0 ? 65536u - (unsigned)(ctas - 1) : 1u);
}

}  // namespace weave
