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
constexpr int kStTokens = 32;                     // one 32-bit mask per expert
constexpr int kStMaxT = 8;                        // largest batch (see stream_slots)
constexpr int kStSlot = 16384;                    // bytes of a ring slot
constexpr int kStMaxSlots = 12, kStMinSlots = 5;
constexpr int kStArea = kStages * kStageBytes + kEpiStageBytes;      // shared memory in front of the SmemTail: ring, then rows
constexpr int kStUnitG = 8, kStUnitD = 16;        // columns of h / of y that one warp works on: 8 gate + 8 up rows, or 16 rows
constexpr int kStWarps = 8;                       // ... so a tile has up to 8 units
constexpr int kStPad = 16;                        // bytes between two rows of x or h in shared memory (no bank conflicts)

// boxes of 1 to 8 units: gate_up as [K/64][gate, up][row][64], down as [K/64][row][64]; 128 of K up to 4 units, 64 from 5 on
struct StreamMaps { CUtensorMap g[kStWarps], d[kStWarps]; };
__host__ __device__ __forceinline__ constexpr int stream_kblocks(int w) { return w <= kStWarps / 2 ? 2 : 1; }

struct StreamShared {      // lies over the SmemTail's segment tables, which this kernel does not use
    uint64_t full[kStMaxSlots], empty[kStMaxSlots];
    uint64_t done[2], freed[2];                   // a tile's stores are issued; its arrival is on its way
    unsigned mask[kMaxEE];                        // bit t: token t selected the expert
    int off[kMaxEE + 1];                          // first row of every expert
    int act[kMaxEE];                              // experts with rows
    int n_act, failed;
    unsigned wsum[8];
    int idx[kStTokens][kMaxTopK], row[kStTokens][kMaxTopK];
    float gate[kStTokens][kMaxTopK];
};
constexpr size_t kStSharedAt = (offsetof(SmemTail, seg_mb0) + 15) / 16 * 16;      // (the tail starts on a 1024-byte boundary)
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

// This CTA's share of a phase: units [u, end) of all active experts' columns, in tiles of 1 to 8 units (equal ones where
// an expert's part is cut) that never span two experts.
struct StreamWalk {
    int u, end, upe;      // upe: units per expert
    int a, c, w;          // the current tile: active expert, first unit in it, units
    __device__ __forceinline__ StreamWalk(int n_act, int upe_, int cta, int ctas) : upe(upe_)
    {
        const int total = n_act * upe_;
        u = (int)((long long)total * cta / ctas);
        end = (int)((long long)total * (cta + 1) / ctas);
    }
    __device__ __forceinline__ bool next()
    {
        if (u >= end) return false;
        a = u / upe;
        c = u - a * upe;
        const int n = min(upe - c, end - u), tiles = (n + kStWarps - 1) / kStWarps;
        w = (n + tiles - 1) / tiles;
        u += w;
        return true;
    }
};

// Top-k of one token by a warp: lane l holds experts l, l + 32, ... as order keys in registers; order, ties and gates as
// in route_block.
__device__ __forceinline__ void stream_route(const KParams &p, StreamShared &X, int t, const float (&lg)[8])
{
    const int lane = threadIdx.x & 31;
    unsigned key[8], bk = 0u;
    int be = 0x7fffffff;
    bool bad = false;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int e = lane + 32 * i;
        float x = lg[i];
        const bool nf = !(fabsf(x) <= 3.402823466e38f);
        bad = bad || (e < p.E && nf);
        x = nf ? -3.402823466e38f : x;
        x = __fadd_rn(x, 0.0f);
        key[i] = e < p.E ? float_order_key(x) : 0u;
        if (key[i] > bk) { bk = key[i]; be = e; }
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicCAS(&p.ctl->status, 0, kErrNonFinite);
    float vmax = 0.f, sum = 0.f, mine = 0.f;
    int my_e = 0;
#pragma unroll 1
    for (int j = 0; j < p.k; ++j) {
        const unsigned top = __reduce_max_sync(0xffffffffu, bk);
        const int hi = (int)__reduce_min_sync(0xffffffffu, bk == top ? (unsigned)be : 0x7fffffffu);
        const float v = float_from_order_key(top);
        if (j == 0) vmax = v;
        const float pj = expf(v - vmax);
        sum += pj;
        if (lane == j) { mine = pj; my_e = hi; }
        if (lane == 0) atomicOr(&X.mask[hi], 1u << t);
        if ((hi & 31) == lane) {
            bk = 0u; be = 0x7fffffff;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (i == (hi >> 5)) key[i] = 0u;
                if (key[i] > bk) { bk = key[i]; be = lane + 32 * i; }
            }
        }
    }
    if (lane < p.k) {
        X.idx[t][lane] = my_e;
        X.gate[t][lane] = __fdiv_rn(mine, sum);
    }
}

// One tile for a warp: 16 weight rows x 8 * NT tokens, KB blocks of 64 of K per ring slot.  a_off: this lane's ldmatrix row in a
// slot, blk: bytes of a block of K in the slot, b_row: this lane's rows of x or h.  The rows' values are fetched before the wait for the slot.
template <int NT, int KB>
__device__ __forceinline__ bool stream_tile(const KParams &p, StreamShared &X, uint32_t ring, int slots, int &slot, uint32_t &ph,
                                            int nk, bool works, uint32_t a_off, uint32_t blk, const uint32_t (&b_row)[4], float (&acc)[NT][4])
{
    const int lane = threadIdx.x & 31;
    const uint32_t sw = (uint32_t)(lane & 7), kh = (uint32_t)(lane >> 4);
    bool ok = true;
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[n][i] = 0.f;
    for (int kk = 0; kk < nk; ++kk) {
        uint32_t b[NT][2][4];
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int i = 0; i < 2; ++i) ldmatrix_x4(b_row[n] + (uint32_t)(kk * (KB * 128) + i * 64), b[n][i]);
        ok = mbar_wait(&X.full[slot], ph, p, 61) && ok;
        if (works) {
            const uint32_t a0 = ring + (uint32_t)(slot * kStSlot) + a_off;
#pragma unroll
            for (int kb = 0; kb < KB; ++kb) {
                uint32_t a[4][4];
#pragma unroll
                for (int s = 0; s < 4; ++s) ldmatrix_x4(a0 + (uint32_t)kb * blk + (((2u * (uint32_t)s + kh) ^ sw) << 4), a[s]);
                if (kb > 0) {
#pragma unroll
                    for (int n = 0; n < NT; ++n)
#pragma unroll
                        for (int i = 0; i < 2; ++i) ldmatrix_x4(b_row[n] + (uint32_t)(kk * (KB * 128) + kb * 128 + i * 64), b[n][i]);
                }
#pragma unroll
                for (int s = 0; s < 4; ++s)
#pragma unroll
                    for (int n = 0; n < NT; ++n) mma_16816(acc[n], a[s], b[n][s >> 1][2 * (s & 1)], b[n][s >> 1][2 * (s & 1) + 1]);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&X.empty[slot]);
        if (++slot == slots) { slot = 0; ph ^= 1u; }
    }
    return ok;
}

__global__ void __launch_bounds__(kStThreads, 1)
weave_stream_kernel(const __grid_constant__ KParams p, const __grid_constant__ StreamMaps tm)
{
    uint8_t *stages = smem_stages();
    SmemTail &S = smem_tail();
    StreamShared &X = *reinterpret_cast<StreamShared *>(reinterpret_cast<uint8_t *>(&S) + kStSharedAt);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int cta = (int)blockIdx.x, ctas = (int)gridDim.x;
    const int slots = p.st_slots;
    const uint32_t ring = smem_u32(stages), rows_s = ring + (uint32_t)(slots * kStSlot);

    // the logits of this warp's tokens and the batch's rows of x start on their way before anything else
    float lg[2][8];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int t = warp + 16 * r;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int e = lane + 32 * i;
            lg[r][i] = t < p.T && e < p.E ? __ldcg(p.logits + (size_t)t * p.E + e) : 0.f;
        }
    }
    const uint32_t pitch_x = (uint32_t)p.H * 2u + kStPad;
    if (warp > 0) {
        const int per_row = p.H >> 3;
        for (int t = 0; t < p.T; ++t)
            for (int c = tid - 32; c < per_row; c += kStThreads - 32)
                cp_async_16(rows_s + (uint32_t)t * pitch_x + (uint32_t)(c * 16), p.x + (size_t)t * p.H + c * 8);
    }
    if (tid == 0) {
        const unsigned odd = (ld_relaxed_u32(&p.ctl->epoch) >> 16) & 1u;
#pragma unroll 1
        for (int i = 0; i < slots; ++i) { mbar_init(&X.full[i], 1); mbar_init(&X.empty[i], kStWarps); }
#pragma unroll 1
        for (int i = 0; i < 2; ++i) { mbar_init(&X.done[i], kStWarps); mbar_init(&X.freed[i], 1); }
        fence_mbar_init();
        S.cs = reinterpret_cast<CtlSet *>(p.sets + (odd ? ctl_set_bytes(p.nmb_max) : 0));
        S.h_ready = reinterpret_cast<unsigned *>(S.cs + 1) + kFine * kMaxEE + p.nmb_max;
        X.failed = 0;
    }
    if (tid < kMaxEE) X.mask[tid] = tid >= p.E && tid < p.EE ? (2u << (p.T - 1)) - 1u : 0u;
    __syncthreads();
    {
        const size_t bytes = ctl_set_bytes(p.nmb_max);
        uint4 *other = reinterpret_cast<uint4 *>(p.sets + (reinterpret_cast<uint8_t *>(S.cs) == p.sets ? bytes : 0));
        for (size_t i = (size_t)cta * kStThreads + tid; i < bytes / 16; i += (size_t)ctas * kStThreads)
            other[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    // ================= routing, counts, offsets, active experts
    if (warp < p.T) stream_route(p, X, warp, lg[0]);
    if (warp + 16 < p.T) stream_route(p, X, warp + 16, lg[1]);
    __syncthreads();
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

    if (warp == 0) {
        // ---------------- producer
        if (lane == 0) {
            int slot = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int phase = 0; phase < 2 && ok; ++phase) {
                StreamWalk wk(A, phase ? p.H / kStUnitD : p.I / kStUnitG, cta, ctas);
                while (ok && wk.next()) {
                    const int e = X.act[wk.a], kb = stream_kblocks(wk.w), nk = (phase ? p.I : p.H) / (64 * kb);
                    const int row = phase ? e * p.H + wk.c * kStUnitD : e * 2 * p.I + wk.c * kStUnitG;
                    const CUtensorMap *map = phase ? &tm.d[wk.w - 1] : &tm.g[wk.w - 1];
                    for (int kk = 0; kk < nk; ++kk) {
                        if (!mbar_wait(&X.empty[slot], ph ^ 1u, p, 60)) { ok = false; break; }
                        mbar_arrive_expect_tx(&X.full[slot], (uint32_t)(wk.w * kb * 2048));
                        const uint32_t dst = ring + (uint32_t)(slot * kStSlot);
                        if (phase) tma_load_3d(dst, map, 0, row, kb * kk, &X.full[slot]);
                        else tma_load_4d(dst, map, 0, row, 0, kb * kk, &X.full[slot]);
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
            // ---------------- a release at GPU scope waits until the tile's stores are performed: not the products' business
            if (lane == 0) {
                int tile = 0;
                bool ok = true;
                for (int phase = 0; phase < 2 && ok; ++phase) {
                    StreamWalk wk(A, phase ? p.H / kStUnitD : p.I / kStUnitG, cta, ctas);
                    for (; ok && wk.next(); ++tile) {
                        ok = mbar_wait(&X.done[tile & 1], (uint32_t)((tile >> 1) & 1), p, 64);
                        if (ok) red_release_add_u32(phase ? &S.cs->y_done[0] : &S.h_ready[wk.a], (unsigned)wk.w);
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
                p.ctl->plan_nmb = A;      // (at most 32 rows per expert: one m-block and one row tile each)
                p.ctl->plan_ngemm = A * (p.nt0 + p.nt1);
            }
            // the dispatched rows, row r by CTA r mod N
            const int P = p.T * (p.k + p.S);
            for (int r = cta + ctas * (warp - 2); r < P; r += ctas * 6) {
                int lo = 0, hi = p.EE;      // largest expert that starts at or before r (empty ones share a start with the next)
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (X.off[mid] <= r) lo = mid; else hi = mid;
                }
                const int t = (int)__fns(X.mask[lo], 0u, r - X.off[lo] + 1);
                const uint4 *src = reinterpret_cast<const uint4 *>(p.x + (size_t)t * p.H);
                uint4 *dst = reinterpret_cast<uint4 *>(p.xe + (size_t)r * p.H);
                for (int c = lane; c < (p.H >> 3); c += 32) dst[c] = __ldg(src + c);
            }
        } else {
            // ---------------- the products
            const int wi = warp - 8;
            int slot = 0, tile = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int phase = 0; phase < 2; ++phase) {
                StreamWalk wk(A, phase ? p.H / kStUnitD : p.I / kStUnitG, cta, ctas);
                const uint32_t pitch = phase ? (uint32_t)p.I * 2u + kStPad : pitch_x;
                int cur = -1;
                for (; wk.next(); ++tile) {
                    const int e = X.act[wk.a], n_e = X.off[e + 1] - X.off[e], row0 = X.off[e];
                    const int nk = (phase ? p.I : p.H) / (64 * stream_kblocks(wk.w));
                    if (phase && wk.a != cur) {
                        // the next expert's rows of h, once all of them are there and nobody reads what they replace
                        cur = wk.a;
                        named_barrier_sync<2, kStWarps * 32>();
                        if (lane == 0) ok = flag_wait_ge(&S.h_ready[wk.a], (unsigned)(p.I / kStUnitG), p, 62) && ok;
                        __syncwarp();
                        const int per_row = p.I >> 3, ctid = tid - 256;
                        const __nv_bfloat16 *src = p.hbuf + (size_t)row0 * p.I;
                        for (int t = 0; t < n_e; ++t)
                            for (int c = ctid; c < per_row; c += kStWarps * 32)
                                cp_async_16(rows_s + (uint32_t)t * pitch + (uint32_t)(c * 16), src + (size_t)t * p.I + c * 8);
                        cp_async_wait_all();
                        named_barrier_sync<2, kStWarps * 32>();
                    }
                    uint32_t b_row[4];
#pragma unroll
                    for (int n = 0; n < 4; ++n) {
                        const int i = 8 * n + (lane & 7);
                        const int r = phase ? (i < n_e ? i : 0) : (int)__fns(X.mask[e], 0u, i < n_e ? i + 1 : 1);
                        b_row[n] = rows_s + (uint32_t)r * pitch + (uint32_t)((lane >> 3) * 16);
                    }
                    const uint32_t half = (uint32_t)((lane >> 3) & 1);      // rows 8..15 of the warp's sixteen
                    const uint32_t a_off = phase ? (uint32_t)(wi * 16 + (lane & 7) + 8 * (int)half) * 128u
                                                 : (uint32_t)(wi * 8 + (lane & 7)) * 128u + half * (uint32_t)(wk.w * 1024);
                    const uint32_t blk = (uint32_t)(wk.w * 2048);
                    const bool works = wi < wk.w;
                    const int col = phase ? wk.c * kStUnitD + wi * 16 + (lane >> 2) : wk.c * kStUnitG + wi * 8 + (lane >> 2);
                    __nv_bfloat16 *dst = phase ? p.y + (size_t)row0 * p.H + col : p.hbuf + (size_t)row0 * p.I + col;
                    const size_t dpitch = phase ? (size_t)p.H : (size_t)p.I;
                    auto run = [&](auto nt, auto kb) {
                        constexpr int NT = decltype(nt)::value;
                        float acc[NT][4];
                        ok = stream_tile<NT, decltype(kb)::value>(p, X, ring, slots, slot, ph, nk, works, a_off, blk, b_row, acc) && ok;
                        if (works) {
#pragma unroll
                            for (int n = 0; n < NT; ++n)
#pragma unroll
                                for (int i = 0; i < 2; ++i) {      // this lane has tokens 2q and 2q + 1 of every eight
                                    const int r = 8 * n + 2 * (lane & 3) + i;
                                    if (r < n_e) {
                                        __nv_bfloat16 *d = dst + (size_t)r * dpitch;
                                        if (phase) { d[0] = __float2bfloat16_rn(acc[n][i]); d[8] = __float2bfloat16_rn(acc[n][2 + i]); }
                                        else d[0] = __float2bfloat16_rn(silu_mul(acc[n][i], acc[n][2 + i]));
                                    }
                                }
                        }
                    };
                    using C1 = std::integral_constant<int, 1>;
                    using C2 = std::integral_constant<int, 2>;
                    using C4 = std::integral_constant<int, 4>;
                    if (wk.w <= kStWarps / 2) { if (n_e <= 8) run(C1(), C2()); else if (n_e <= 16) run(C2(), C2()); else run(C4(), C2()); }
                    else { if (n_e <= 8) run(C1(), C1()); else if (n_e <= 16) run(C2(), C1()); else run(C4(), C1()); }
                    __syncwarp();
                    if (lane == 0) {
                        if (tile >= 2) ok = mbar_wait(&X.freed[tile & 1], (uint32_t)(((tile >> 1) - 1) & 1), p, 65) && ok;
                        mbar_arrive(&X.done[tile & 1]);
                    }
                }
            }
            if (!ok) X.failed = 1;
        }
    }

    // ================= combine: out[t] = sum over the slots, in slot order, then the shared experts
    __syncthreads();
    if (tid == 0 && !flag_wait_ge(&S.cs->y_done[0], (unsigned)(A * (p.H / kStUnitD)), p, 63)) X.failed = 1;
    __syncthreads();
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
    if (tid == 0) atomicAdd(&p.ctl->epoch, cta == 0 ? 65536u - (unsigned)(ctas - 1) : 1u);
}

}  // namespace weave
