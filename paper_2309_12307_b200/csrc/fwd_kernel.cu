// S2-Attn forward for sm_100a.
//
// A work item is a pair of neighbouring 128-row query tiles of one (batch, head, group): steps "roll",
// "group", "attention" and "roll back" of Algorithm 1 collapse into the choice of TMA coordinates.  Query
// tile i of rolled group g in a head with shift s covers the ORIGINAL tokens given by tile_ref():
// a group is one run of original tokens starting at (g*G + s) mod N, or, where it wraps past the
// sequence end, two runs ([N-G/2, N) followed by [0, G/2) in Algorithm 1), and each run is tiled from
// its own start, so a tile never straddles the sequence end.  Its keys are tiles 0..i of the same
// group, fetched at their own original positions.  When G or s is not a multiple of 128 the last
// tile of a run has fewer than 128 valid rows: the rest of the box holds neighbouring tokens (or
// zero fill), masked as key columns and not stored as query rows.  Outputs are stored at the
// original token rows, which is the roll back.
//
// One persistent block per SM, 512 threads:
//   warps 0-3, 4-7   softmax, two groups that take the tiles of an item in turn (group_of_tile): one thread per
//                    score row, the row's 128 scores in registers (one trip to tensor memory per key tile, no
//                    exchange between threads)
//   warps 8-11       epilogue: O / l -> bf16 -> shared memory -> TMA store (or row stores, ragged tiles)
//   warp 12          work items (cluster launch control: a block takes over blocks that were not launched
//                    yet, heaviest first) and TMA loads, running ahead across items
//   warps 13, 14     tcgen05 MMAs: the score products S = Q K_j^T of both tiles in turn / the products O += P V_j
// (what belongs to a tile's softmax - Q, P, O, statistics, barriers - is kept by group of warps, not by tile)
// While one tile's scores are in the softmax, the tensor cores work for the other tile; K and V tiles
// are fetched once for the 256 query rows, which halves their L2 and shared-memory traffic.
// The scores of a step are in registers 150 clocks after they are complete, and P has tensor memory columns of
// its own, so a tile's next scores are computed while its softmax works on the present ones.  (With P over S the
// chain scores -> softmax -> P V -> next scores of a tile, about 3700 clocks for a step of either tile, was what
// bounded the kernel, with the special-function unit and the tensor pipe each busy half of the time.)
// Tensor memory: O of either tile, P of either tile, then one score buffer (HD = 128) or two.
//
// The last work items of a launch decide how long it takes, so blocks ask for the next one late (when they
// have issued their loads), and one thread decodes it for all warps.  Asking an item ahead and decoding it in
// every warp with 64-bit divisions cost 86 against 73 us on 4 x 2048 tokens with groups of 512, 101 against 80
// on a grouped-query shape (2 x 4096, groups of 1024, head size 64), 2 % on Llama2-7B 32k.
//
// What bounds it: the softmax (a step of both tiles keeps the special-function unit busy for 2048 clocks and the
// tensor pipe for 2048) and, sustained, the power limit: a loop of forward calls on Llama2-7B 32k runs at 1244 TFLOP/s,
// 0.92 of what the cuBLAS loop sustains, the forward within a training step at 1176, 0.84.  Microseconds a call in a
// loop: first form (one query tile per block, two blocks per SM, two threads per row, scores read twice), two tiles with
// P over S, P in columns of its own:
//   Llama2-7B 32k 2383, 1982, 1768; 8k 211, 162, 145; causal 8k 610, 497, 449;
//   groups of 512 99, 73, 70; groups of 200 (head size 64) 40, 32, 29; head size 64 at 32k 1800, 1514, 1374
// Since then the groups of softmax warps take the tiles in turn and the read-out is one loop body; thousands of clocks a
// launch (microseconds follow the clock of the day), before and now:
//   32k 2503, 2484; 8k 213, 204; causal 8k 654, 652; groups of 512 112, 99; groups of 200 (head size 64) 50.5, 47.3;
//   2 x 4096 grouped query 124, 117.5; head size 64 at 32k 2425, 2418
#include "s2a_params.h"
#include "sm100_ptx.cuh"

namespace s2a {

namespace {

template <int HD>
struct FwdCfg {
    static constexpr int kThreads = 512;
    static constexpr int kBoxes = HD / 64;                  // 64-column TMA boxes per tile
    static constexpr int kBoxBytes = kTile * 128;           // 128 rows x 128 bytes
    static constexpr int kTileBytes = kBoxes * kBoxBytes;   // one Q, K, V or O tile
    static constexpr int kRing = (HD == 128) ? 4 : 8;       // K and V tiles in flight: K_0 V_0 K_1 V_1 ...
    static constexpr int kStatBytes = 2 * 2 * kTile * 4;     // row statistics handed to the epilogue
    static constexpr int kBarBytes = 1024 + kStatBytes;
    static constexpr int kSmemBytes = (2 + kRing + 1) * kTileBytes + kBarBytes;
    // Tensor memory columns: O of either tile, P of either tile (bf16, 64 columns), scores.  The scores of a step are
    // in registers soon after they are complete, so for HD = 128, where O takes half of the columns, one
    // score buffer serves both tiles in turn.
    static constexpr int kTmemCols = 512;
    static constexpr int kColO = 0, kColP = 2 * HD, kColS = 2 * HD + 2 * 64;
    static constexpr int kScoreBufs = (HD == 128) ? 1 : 2;
    static_assert(kColS + kScoreBufs * kTile <= kTmemCols, "tensor memory");
    // registers per thread after the split; the launch gives kRegsLaunch to each of the 512
    static constexpr int kRegsLaunch = 128, kRegsSoftmax = 192, kRegsEpilogue = 80, kRegsIssue = 48;
    static_assert(2 * kRegsSoftmax + kRegsEpilogue + kRegsIssue <= 4 * kRegsLaunch, "register split");
};

// Items in flight.  When the producer writes item k, V of item k - 1 has been requested, so the P.V products of the item
// kRing / 2 before that one are done (single tiles, the shortest items, take two slots of the ring each), so the read-out of the
// item that the same group of softmax warps had before, at most two earlier, is done.  Every other warp is further on than the
// read-out.  A group of softmax warps has no part in an item whose only tile (the last pair of an odd number of tiles, single
// tiles) is the other group's, but never misses two in a row; each group walks a list of its own, of the items it has a tile of.
constexpr int kSched = 8;

struct FwdItem {
    int b, h;
    GroupLayout L;
    TilePair t;
};
// The later tile of a pair attends one key tile more than the other one, and it is the only tile where an item has one.
// The two groups of softmax warps take it in turn, from one item of the block to the next: bound to the tiles, one group has
// nothing to do where items are single tiles.  Thousands of clocks a launch, bound and in turn: groups of 128 192 and 175, at
// head size 64 176 and 152; groups of 384 at head size 64 168 and 155; pairs of tiles alone the same to 1 % (8k 204 and 204,
// 32k 2491 and 2506, 2 x 4096 grouped query 118 and 118).  Ragged pairs and a single tile at head size 128 are faster bound
// (groups of 384 173 and 181, of 600 336 and 353), but only where the binding is known when the kernel is compiled: a flag in
// the item that has the groups change places behind single tiles alone is slower than either (186, 365; 8k 208).
__device__ __forceinline__ int group_of_tile(int item, int t) { return (item & 1) ^ t ^ 1; }
__device__ __forceinline__ int tile_of_group(int item, int group) { return (item & 1) ^ group ^ 1; }
struct FwdBars {
    // by group of softmax warps
    uint64_t q_full[2], q_empty[2];
    uint64_t s_full[2];              // S of a tile's step is in tensor memory
    uint64_t s_empty[2];             // a score buffer has been read into registers
    uint64_t p_full[2];              // P of keys [0, 96) of the step is in tensor memory (and O is rescaled)
    uint64_t p_rest[2];              // the other 32 keys
    uint64_t p_empty[2];             // the P.V product of the step is done: P and O may be written
    uint64_t o_full[2], o_empty[2];  // an item's O is complete / has been read out
    uint64_t stat_full[2], stat_empty[2];
    uint64_t kv_full[8], kv_empty[8];
    uint64_t sched_full[kSched];
    uint64_t list_full[2][kSched];   // the same for either group of softmax warps: items that it has a tile of
    uint64_t clc, drain[2];
    alignas(16) uint8_t clc_resp[16];
    FwdItem item[kSched];  // b = -1: no more items
    uint8_t list_slot[2][kSched];  // where the items counted on list_full are
    uint32_t tmem_slot;
    int abort_flag;
};
static_assert(kSched % 2 == 0, "a slot's parity is its item's");
static_assert(kSched >= FwdCfg<64>::kRing / 2 + 3 && kSched >= FwdCfg<128>::kRing / 2 + 3, "an item's slot is free when it is written again");
static_assert(sizeof(FwdBars) <= 1024, "barrier block");

// Threshold (in log2 units) below which a larger running maximum is ignored: P then grows by at
// most 2^8, which bf16 and the fp32 row sum absorb, and O needs no rescale.
constexpr float kLazyRescale = 8.0f;

// The key tiles lie in shared memory with the two middle ones of every four keys exchanged (the tensor map's doing), so
// that a score row's columns are the keys 0 2 1 3, 4 6 5 7, ...  The row sum adds neighbouring keys first (0 + 1, 2 + 3), then
// every fourth of these pairs in one chain, for each half of the tile: with this order of the columns both are packed
// additions of registers that lie side by side.  One chain for all columns of a parity needs no exchange, but leaves lse
// further from its value in 64 bits (relative error, Llama2-7B 16k 4.69e-8 instead of 4.61e-8, 100,000 tokens 4.43e-8
// instead of 4.31e-8) in the same time: 32k 1883 and 1862 us, 8k 155 and 155, head size 64 at 16k 385 and 389, 2 x 4096
// tokens grouped query 67.4 and 67.9.  The pairs as scalar additions take 1926, 156, 391 and 70.5.
__device__ __forceinline__ constexpr int key_of_column(int x) { return (x & ~3) | ((x & 1) << 1) | ((x >> 1) & 1); }

// Work item `id`; false marks a slot of a group that has fewer pairs than the largest one.
__device__ __forceinline__ bool fwd_item(const FwdParams& p, int id, FwdItem* w) {
    int unit, rank, g;
    p.order.decode(id, &unit, &rank);
    w->b = p.by_heads(p.geo.by_groups(unit, &g), &w->h);
    w->L = group_layout(p.geo, (w->h < p.geo.n_unshifted) ? 0 : p.geo.shift, g);
    if (rank >= pairs_of_group(w->L, p.single)) return false;
    w->t = tile_pair(w->L, rank, p.single);
    return true;
}

template <int HD>
__global__ void __launch_bounds__(FwdCfg<HD>::kThreads, 1) s2a_fwd_kernel(const __grid_constant__ FwdParams p) {
    using C = FwdCfg<HD>;
    extern __shared__ __align__(1024) uint8_t smem[];  // 1024-byte aligned: checked below
    uint8_t* sQ = smem;                                // two query tiles
    uint8_t* sKV = sQ + 2 * C::kTileBytes;             // ring of K and V tiles
    uint8_t* sO = sKV + C::kRing * C::kTileBytes;      // one output tile on its way out
    FwdBars* bars = reinterpret_cast<FwdBars*>(sO + C::kTileBytes);
    float* sStat = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + 1024);  // [group][m, l][128 rows]

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int t = 0; t < 2; ++t) {
            // hand-offs by four warps count one arrival per warp: 128 arrivals are 128 updates of one word of
            // shared memory, whose bandwidth the operand reads of the MMAs need
            mbar_init(&bars->q_full[t], 1);
            mbar_init(&bars->q_empty[t], 1);
            mbar_init(&bars->s_full[t], 1);
            mbar_init(&bars->s_empty[t], 4);
            mbar_init(&bars->p_empty[t], 1);
            mbar_init(&bars->p_full[t], 4);
            mbar_init(&bars->p_rest[t], 4);
            mbar_init(&bars->o_full[t], 1);
            mbar_init(&bars->o_empty[t], 4);
            mbar_init(&bars->stat_full[t], 4);
            mbar_init(&bars->stat_empty[t], 4);
            mbar_init(&bars->drain[t], 1);
        }
        for (int x = 0; x < C::kRing; ++x) {
            mbar_init(&bars->kv_full[x], 1);
            mbar_init(&bars->kv_empty[x], 1);
        }
        for (int x = 0; x < kSched; ++x) {
            mbar_init(&bars->sched_full[x], 1);
            mbar_init(&bars->list_full[0][x], 1);
            mbar_init(&bars->list_full[1][x], 1);
        }
        mbar_init(&bars->clc, 1);
        fence_barrier_init();
        tma_prefetch_desc(&p.tm_q);
        tma_prefetch_desc(&p.tm_k);
        tma_prefetch_desc(&p.tm_v);
        tma_prefetch_desc(&p.tm_o);
    }
    if (warp == 13) {
        tmem_alloc(&bars->tmem_slot, C::kTmemCols);
        tmem_relinquish();
    }
    wait_for_predecessor();
    // A bounded wait that expired earlier (in any kernel) leaves the status word set: later blocks
    // then return at once instead of each running into its own time limit.
    if (threadIdx.x == 0) {
        int bad = *reinterpret_cast<volatile int*>(p.status);
        if ((smem_u32(smem) & 1023u) != 0) {  // cannot happen: nothing precedes the dynamic array
            bad = kWaitFwd + 99;
            atomicCAS(p.status, 0, bad);
            *reinterpret_cast<volatile int*>(p.host_status) = bad;
        }
        bars->abort_flag = bad;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    release_successor();
    const uint32_t tmem_base = bars->tmem_slot;
    if (bars->abort_flag != 0) {
        if (warp == 13) tmem_dealloc(tmem_base, C::kTmemCols);
        return;
    }
    const WaitCtx ctx{&bars->abort_flag, p.status, p.host_status};

    // Every consumer warp walks the same sequence of items, as the scheduling thread has decoded them (the
    // divisions of fwd_item cost a warp about a thousand clocks): the k-th one, false = the end (or aborting).
    auto next_item = [&](int k, int where, FwdItem* w) -> bool {
        if (!mbar_wait_uniform(&bars->sched_full[k % kSched], (k / kSched) & 1, ctx, where)) return false;
        *w = bars->item[k % kSched];
        return w->b >= 0;
    };

    if (warp >= 12) {
        setmaxnreg_dec<C::kRegsIssue>();
        if (warp == 12) {
            // ======================= work items, TMA loads ===========================================
            if (lane == 0) {
                uint32_t kv = 0;              // K and V tiles requested so far
                uint32_t n_q[2] = {0, 0};     // query tiles requested so far for either group
                bool ok = true;
                ItemSource items{&bars->clc, bars->clc_resp};
                int id = static_cast<int>(blockIdx.x);
                uint32_t n_list[2] = {0, 0};  // items in the list of either group
                auto load_q = [&](const FwdItem& w, int t, int g) {
                    const uint32_t n = g ? n_q[1]++ : n_q[0]++;
                    if (!mbar_wait(&bars->q_empty[g], (n & 1) ^ 1, ctx, kWaitFwd + 2)) {
                        --(g ? n_q[1] : n_q[0]);
                        ok = false;
                        return;
                    }
                    mbar_expect_tx(&bars->q_full[g], C::kTileBytes);
                    const int tok0 = tile_ref(w.L, t ? w.t.i[1] : w.t.i[0]).tok0;
                    for (int bx = 0; bx < C::kBoxes; ++bx)
                        tma_load_4d(sQ + g * C::kTileBytes + bx * C::kBoxBytes, &p.tm_q, &bars->q_full[g], bx * 64, w.h, tok0, w.b);
                };
                auto enlist = [&](int k, int g) {
                    const uint32_t n = g ? n_list[1]++ : n_list[0]++;
                    bars->list_slot[g][n % kSched] = static_cast<uint8_t>(k % kSched);
                    mbar_arrive(&bars->list_full[g][n % kSched]);
                };
                auto load_kv = [&](const FwdItem& w, int hk, bool k_tile, int tok0) {
                    const int st = kv % C::kRing;
                    if (!mbar_wait(&bars->kv_empty[st], ((kv / C::kRing) & 1) ^ 1, ctx, kWaitFwd + 3)) { ok = false; return; }
                    mbar_expect_tx(&bars->kv_full[st], C::kTileBytes);
                    for (int bx = 0; bx < C::kBoxes; ++bx) {
                        uint8_t* dst = sKV + st * C::kTileBytes + bx * C::kBoxBytes;
                        if (k_tile) tma_load_5d(dst, &p.tm_k, &bars->kv_full[st], hk * HD + bx * 64, 0, 0, tok0 / 4, w.b);
                        else tma_load_4d(dst, &p.tm_v, &bars->kv_full[st], bx * 64, hk, tok0, w.b);
                    }
                    ++kv;
                };
                for (int k = 0; ok; ++k) {
                    // A copy of its own: read back from shared memory for every load, it holds the loads up (Llama2-7B 8k 214,600
                    // against 209,300 clocks a launch, 4 x 8192 806,800 against 790,200, groups of 600 406,300 against 398,300,
                    // 64-wide heads in groups of 128 170,500 against 161,700), although the copy costs a few registers too many.
                    FwdItem w;
                    while (id >= 0 && !fwd_item(p, id, &w)) {  // skip the empty slots of smaller groups
                        id = items.next(ctx, kWaitFwd + 1, &ok);
                    }
                    if (id < 0) w.b = -1;
                    bars->item[k % kSched] = w;
                    mbar_arrive(&bars->sched_full[k % kSched]);  // release: the item is visible to whoever sees the phase
                    const int g1 = group_of_tile(k, 1), g0 = group_of_tile(k, 0);
                    enlist(k, g1);
                    if (id < 0 || w.t.n[0] > 0) enlist(k, g0);
                    if (id < 0) break;
                    const int hk = p.geo.by_rep(w.h);
                    for (int j = 0; ok && j < w.t.n[1]; ++j) {
                        const int tok0 = tile_ref(w.L, w.t.j_begin + j).tok0;
                        load_kv(w, hk, true, tok0);
                        if (j == 0 && ok) load_q(w, 1, g1);
                        if (j == 0 && ok && w.t.n[0] > 0) load_q(w, 0, g0);
                        if (ok) load_kv(w, hk, false, tok0);
                    }
                    if (ok) id = items.next(ctx, kWaitFwd + 1, &ok);
                }
                // nothing may land after the block has gone
                if (bars->abort_flag != 0) {
                    for (int t = 0; t < 2; ++t)
                        if (n_q[t] > 0) mbar_wait_drain(&bars->q_full[t], (n_q[t] - 1) & 1);
                    for (uint32_t x = (kv > C::kRing ? kv - C::kRing : 0); x < kv; ++x)
                        mbar_wait_drain(&bars->kv_full[x % C::kRing], (x / C::kRing) & 1);
                }
            }
            __syncwarp();
        } else if (warp <= 14) {
            // ======================= MMA issuers: warp 13 for S = Q K^T, warp 14 for O += P V ============
            // The whole warp walks the loop so that addresses and descriptors stay warp-uniform values;
            // only the MMA and commit instructions themselves are issued by one elected lane.  Both take the
            // tiles in turn: tile 1, tile 0 of key tile j, then of j + 1 (tile 0 has no products with the
            // last key tile), so that the groups of softmax warps are served in turn across items as well (tile 0 first:
            // 8k 204,000 -> 211,000 clocks a launch, 2 x 4096 grouped query 118,000 -> 129,500).
            // K tiles are in the even slots of the ring, V tiles in the odd ones.
            constexpr uint32_t idesc_s = idesc_bf16(128, kTile, 0, 0);  // S = Q K^T   (both K-major)
            constexpr uint32_t idesc_o = idesc_bf16(128, HD, 0, 1);     // O += P V    (V is MN-major)
            const bool is_s = warp == 13;
            const uint32_t aKV = smem_u32(sKV), dQ0 = desc_lo_k_major(smem_u32(sQ));
            uint32_t kv = 0;                    // ring position of the item's K_0
            uint32_t n_it[2] = {0, 0};          // items of either group so far
            uint32_t n_st[2] = {0, 0}, n_s = 0; // steps of either group, score products
            bool ok = true;
            for (int k = 0; ok; ++k) {
                FwdItem w;
                if (!next_item(k, kWaitFwd + 10, &w)) break;
                const int n1 = w.t.n[1], n0 = w.t.n[0];
#pragma unroll 1
                for (int h = 0; ok && h < 2 * n1; ++h) {
                    const int t = (h & 1) ^ 1, j = h >> 1, n = t ? n1 : n0, g = group_of_tile(k, t);
                    if (j >= n) continue;
                    const uint32_t x = kv + 2 * j + (is_s ? 0 : 1);
                    const bool last_use = t == 0 || j >= n0;  // of this K or V tile
                    const uint32_t st = (g ? n_st[1] : n_st[0]) & 1, it = (g ? n_it[1] : n_it[0]) & 1;
                    // what tile 1 has used, tile 0 need not wait for again
                    if (t == 1 && !mbar_wait_uniform(&bars->kv_full[x % C::kRing], (x / C::kRing) & 1, ctx, kWaitFwd + 5)) { ok = false; break; }
                    if (is_s) {
                        if (j == 0 && !mbar_wait_uniform(&bars->q_full[g], it, ctx, kWaitFwd + 4)) { ok = false; break; }
                        const int buf = C::kScoreBufs == 1 ? 0 : g;
                        const uint32_t use = C::kScoreBufs == 1 ? n_s & 1 : st;
                        if (!mbar_wait_uniform(&bars->s_empty[buf], use ^ 1, ctx, kWaitFwd + 6)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t at_g = dQ0 + g * (C::kTileBytes >> 4);
                        const uint32_t at_x = desc_lo_k_major(aKV + (x % C::kRing) * C::kTileBytes);
                        const uint32_t acc = tmem_base + C::kColS + buf * kTile;
                        if (elect_one()) {
#pragma unroll
                            for (int kk = 0; kk < HD / 16; ++kk)
                                mma_ss(acc, at_g + desc_step_k_major(kk, C::kBoxBytes), at_x + desc_step_k_major(kk, C::kBoxBytes), idesc_s, kk > 0);
                            mma_commit(&bars->s_full[g]);
                            if (last_use) mma_commit(&bars->kv_empty[x % C::kRing]);
                            if (j == n - 1) mma_commit(&bars->q_empty[g]);
                        }
                        __syncwarp();
                        ++n_s;
                    } else {
                        if (j == 0 && !mbar_wait_uniform(&bars->o_empty[g], it ^ 1, ctx, kWaitFwd + 7)) { ok = false; break; }
                        const uint32_t at_x = desc_lo_mn_major(aKV + (x % C::kRing) * C::kTileBytes, C::kBoxBytes);
                        const uint32_t at_g = tmem_base + C::kColP + g * 64, acc = tmem_base + C::kColO + g * HD;
                        if (!mbar_wait_uniform(&bars->p_full[g], st, ctx, kWaitFwd + 8)) { ok = false; break; }
                        tc_fence_after();
                        if (elect_one()) {
#pragma unroll
                            for (int kk = 0; kk < 6; ++kk) mma_ts(acc, at_g + kk * 8, at_x + kk * kDescStepMn, idesc_o, (j > 0) || (kk > 0));
                        }
                        __syncwarp();
                        if (!mbar_wait_uniform(&bars->p_rest[g], st, ctx, kWaitFwd + 9)) { ok = false; break; }
                        tc_fence_after();
                        if (elect_one()) {
#pragma unroll
                            for (int kk = 6; kk < 8; ++kk) mma_ts(acc, at_g + kk * 8, at_x + kk * kDescStepMn, idesc_o, 1);
                            mma_commit(&bars->p_empty[g]);
                            if (last_use) mma_commit(&bars->kv_empty[x % C::kRing]);
                            if (j == n - 1) mma_commit(&bars->o_full[g]);
                        }
                        __syncwarp();
                    }
                    if (g) ++n_st[1], n_it[1] += j == n - 1;
                    else ++n_st[0], n_it[0] += j == n - 1;
                }
                kv += 2 * n1;
            }
            // MMAs already issued must finish before tensor memory is released
            if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&bars->abort_flag) != 0)) {
                if (elect_one()) {
                    mma_commit(&bars->drain[is_s]);
                    mbar_wait_drain(&bars->drain[is_s], 0);
                }
            }
            __syncwarp();
        }
    } else if (warp >= 8) {
        // =========================== epilogue ========================================================
        setmaxnreg_dec<C::kRegsEpilogue>();
        const int quad = warp & 3;
        const int row = quad * 32 + lane;
        const uint32_t t_row = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
        uint32_t n_o[2] = {0, 0};
        bool ok = true;
        for (int k = 0; ok; ++k) {
            FwdItem w;
            // the four warps leave together, or the ones that stay would wait for the others below
            if (!named_barrier_and(1, 128, next_item(k, kWaitFwd + 11, &w))) break;
            // One loop body for both tiles and all columns: what the read-out adds to the code that the softmax warps run beside
            // costs more than its branches.  Clocks a launch with the tiles written out twice at head size 128 and all columns
            // written out, and like this: groups of 200 114,800 and 100,000, of 384 211,900 and 180,200, of 600 398,400 and
            // 351,400, Llama2-7B 8k 208,400 and 204,300, 32k 2,508,000 and 2,502,000; head size 64, groups of 384 161,800 and
            // 154,300, 32k 2,440,000 and 2,420,000.
#pragma unroll 1
            for (int t = 0; t < 2; ++t) {
                if ((t ? w.t.n[1] : w.t.n[0]) == 0) continue;
                const int g = group_of_tile(k, t);
                const TileRef tq = tile_ref(w.L, t ? w.t.i[1] : w.t.i[0]);
                const uint32_t n_done = g ? n_o[1]++ : n_o[0]++;
                const bool whole = tq.valid == kTile;
                // the tile stored last must have left the staging buffer (thread 0 of the four warps stores)
                if (threadIdx.x == 256) bulk_wait_read<0>();
                ok = mbar_wait_uniform(&bars->stat_full[g], n_done & 1, ctx, kWaitFwd + 12) &&
                     mbar_wait_uniform(&bars->o_full[g], n_done & 1, ctx, kWaitFwd + 13);
                ok = named_barrier_and(1, 128, ok);
                if (!ok) break;
                tc_fence_after();
                const float m = sStat[g * 256 + row], l = sStat[g * 256 + 128 + row];
                mbar_arrive_warp(&bars->stat_empty[g]);
                const float inv_l = 1.0f / l;
                const int tok = tq.tok0 + row;
                const bool row_valid = row < tq.valid;  // rows past the end of a ragged tile are not part of the group
                __nv_bfloat16* orow = p.o + ((static_cast<size_t>(w.b) * p.geo.N + tok) * p.geo.H + w.h) * HD;
#pragma unroll 1
                for (int c = 0; c < HD / 32; ++c) {
                    uint32_t r[32];
                    tmem_ld_32x32(t_row + C::kColO + g * HD + c * 32, r);
                    tmem_wait_ld();
                    const uint32_t dst_s = smem_u32(sO) + (c >> 1) * C::kBoxBytes + row * 128;
                    uint4* dst_g = reinterpret_cast<uint4*>(orow + c * 32);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        uint4 pk;
                        pk.x = pack_bf16(__uint_as_float(r[8 * e + 0]) * inv_l, __uint_as_float(r[8 * e + 1]) * inv_l);
                        pk.y = pack_bf16(__uint_as_float(r[8 * e + 2]) * inv_l, __uint_as_float(r[8 * e + 3]) * inv_l);
                        pk.z = pack_bf16(__uint_as_float(r[8 * e + 4]) * inv_l, __uint_as_float(r[8 * e + 5]) * inv_l);
                        pk.w = pack_bf16(__uint_as_float(r[8 * e + 6]) * inv_l, __uint_as_float(r[8 * e + 7]) * inv_l);
                        if (whole) {
                            // 16-byte chunk (4 (c & 1) + e) of the 128-byte row, swizzled as the tensor map has it
                            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst_s + (((4 * (c & 1) + e) ^ (row & 7)) << 4)),
                                         "r"(pk.x), "r"(pk.y), "r"(pk.z), "r"(pk.w)
                                         : "memory");
                        } else if (row_valid) {
                            dst_g[e] = pk;
                        }
                    }
                }
                tc_fence_before();
                mbar_arrive_warp(&bars->o_empty[g]);
                if (whole) {
                    fence_proxy_async();
                    named_barrier(1, 128);
                    if (threadIdx.x == 256) {
                        for (int bx = 0; bx < C::kBoxes; ++bx)
                            tma_store_4d(&p.tm_o, sO + bx * C::kBoxBytes, bx * 64, w.h, tq.tok0, w.b);
                        bulk_commit_group();
                    }
                }
                // natural-log sum-exp of the scaled scores
                if (row_valid) p.lse[(static_cast<size_t>(w.b) * p.geo.H + w.h) * p.geo.N + tok] = (m + log2f(l)) * 0.6931471805599453f;
            }
        }
        if (threadIdx.x == 256) bulk_wait_all();
    } else {
        // =========================== softmax =========================================================
        setmaxnreg_inc<C::kRegsSoftmax>();
        // This warp's group takes a tile of every item, or of every other one.  Known to the compiler as the same for the whole
        // warp, it takes 0.8 % off long groups at head size 128 (32k 2,505,000 -> 2,484,000 clocks a launch, causal 8k 657,000
        // -> 652,000, groups of 384 180,500 -> 177,500) and adds 1 % at 64 (causal 8k 622,600 -> 630,300).
        const int group = HD == 128 ? __shfl_sync(0xffffffffu, warp >> 2, 0) : warp >> 2;
        const int quad = warp & 3;             // tensor-memory lane quadrant this warp may access
        const int row = quad * 32 + lane;
        const uint32_t t_row = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
        const uint32_t tS = t_row + C::kColS + (C::kScoreBufs == 1 ? 0 : group * kTile), tP = t_row + C::kColP + group * 64;
        const float c2 = p.scale_log2;
        const uint64_t c2x2 = f2_pack(c2, c2);
        uint32_t n_s = 0, n_it = 0;
        bool ok = true;
        for (int k = 0; ok; ++k) {
            if (!mbar_wait_uniform(&bars->list_full[group][k % kSched], (k / kSched) & 1, ctx, kWaitFwd + 14)) break;
            const int slot = bars->list_slot[group][k % kSched];
            const FwdItem w = bars->item[slot];
            if (w.b < 0) break;
            const int n = tile_of_group(slot, group) ? w.t.n[1] : w.t.n[0];
            float m_used = 0.f;   // running maximum in use, scaled to log2 units
            // running sum of exp2(s*c2 - m_used) over the keys [0, 64) and [64, 128) of the tiles
            float l[2] = {0.f, 0.f};
            for (int j = 0; j < n; ++j, ++n_s) {
                const int k_valid = tile_ref(w.L, w.t.j_begin + j).valid;
                if (!mbar_wait_uniform(&bars->s_full[group], n_s & 1, ctx, kWaitFwd + 15)) { ok = false; break; }
                tc_fence_after();
                uint32_t s[4][32];
                tmem_ld_32x32(tS, s[0]);
                tmem_ld_32x32(tS + 32, s[1]);
                tmem_ld_32x32(tS + 64, s[2]);
                tmem_ld_32x32(tS + 96, s[3]);
                tmem_wait_ld();
                tc_fence_before();
                mbar_arrive_warp(&bars->s_empty[C::kScoreBufs == 1 ? 0 : group]);
                // Key x of the tile is visible to query row r iff it is one of the tile's valid rows and,
                // on the diagonal tile, x <= r.  Off the diagonal a full tile needs no mask at all.
                const bool last = (j == n - 1);
                if (last || k_valid < kTile) {
                    const int vis = (last && row < k_valid) ? row : k_valid - 1;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (c * 32 + key_of_column(e) > vis) s[c][e] = 0xff800000u;  // -inf
                }
                float mx4[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    mx4[c] = fmaxf(__uint_as_float(s[c][0]), __uint_as_float(s[c][1]));
#pragma unroll
                    for (int e = 2; e < 32; e += 2) mx4[c] = fmax3(mx4[c], __uint_as_float(s[c][e]), __uint_as_float(s[c][e + 1]));
                }
                const float m_new = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * c2;
                // the P.V product of this tile's step before is done: P and O may be written
                if (n_s > 0 && !mbar_wait_uniform(&bars->p_empty[group], (n_s - 1) & 1, ctx, kWaitFwd + 17)) { ok = false; break; }
                tc_fence_after();
                if (j == 0) {
                    m_used = m_new;
                } else {
                    const bool need = (m_new - m_used) > kLazyRescale;
                    if (__any_sync(0xffffffffu, need)) {
                        const float alpha = need ? fast_exp2(m_used - m_new) : 1.0f;
                        l[0] *= alpha, l[1] *= alpha;
#pragma unroll 1
                        for (int c = 0; c < HD / 16; ++c) {
                            uint32_t o[16];
                            const uint32_t t_o = t_row + C::kColO + group * HD + c * 16;
                            tmem_ld_32x16(t_o, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                            tmem_st_32x16(t_o, o);
                        }
                        if (need) m_used = m_new;
                    }
                }
                const uint64_t nm = f2_pack(-m_used, -m_used);
                uint64_t sum[2];  // of a half of the tile: chains 0 and 1, chains 2 and 3 (see key_of_column)
                auto add_chunk = [&](int c) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        auto weight = [&](int x) { return __uint_as_float(s[c][4 * e + x]); };
                        const uint64_t pairs = f2_add(f2_pack(weight(0), weight(1)), f2_pack(weight(2), weight(3)));
                        sum[e & 1] = (c & 1) == 0 && e < 2 ? pairs : f2_add(sum[e & 1], pairs);
                    }
                    if (c & 1) {
                        float a0, a1, b0, b1;
                        f2_unpack(sum[0], a0, a1);
                        f2_unpack(sum[1], b0, b1);
                        l[c >> 1] += (a0 + a1) + (b0 + b1);
                    }
                };
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t pk[16];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        float p0, p1, p2, p3;  // weights of the keys 4 e to 4 e + 3
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(s[c][4 * e]), __uint_as_float(s[c][4 * e + 1])), c2x2, nm), p0, p2);
                        f2_unpack(f2_fma(f2_pack(__uint_as_float(s[c][4 * e + 2]), __uint_as_float(s[c][4 * e + 3])), c2x2, nm), p1, p3);
                        p0 = fast_exp2(p0), p1 = fast_exp2(p1), p2 = fast_exp2(p2), p3 = fast_exp2(p3);
                        s[c][4 * e] = __float_as_uint(p0), s[c][4 * e + 1] = __float_as_uint(p2);
                        s[c][4 * e + 2] = __float_as_uint(p1), s[c][4 * e + 3] = __float_as_uint(p3);
                        pk[2 * e] = pack_bf16(p0, p1), pk[2 * e + 1] = pack_bf16(p2, p3);
                    }
                    tmem_st_32x16(tP + c * 16, pk);
                    if (c >= 2) {
                        tmem_wait_st();
                        tc_fence_before();
                        mbar_arrive_warp(c == 2 ? &bars->p_full[group] : &bars->p_rest[group]);
                    }
                    // the sum of a chunk beside the exponentials of the next: all sums at the end cost 2 % (head size 64, 16k)
                    if (c > 0) add_chunk(c - 1);
                    if (c == 3) add_chunk(3);
                }
            }
            if (!ok || !mbar_wait_uniform(&bars->stat_empty[group], (n_it & 1) ^ 1, ctx, kWaitFwd + 16)) break;
            ++n_it;
            sStat[group * 256 + row] = m_used;
            sStat[group * 256 + 128 + row] = l[0] + l[1];
            mbar_arrive_warp(&bars->stat_full[group]);
        }
    }

    // ---- teardown ------------------------------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    if (warp == 13) {
        tc_fence_after();
        tmem_dealloc(tmem_base, C::kTmemCols);
    }
}

template <int HD>
cudaError_t configure_one() {
    using C = FwdCfg<HD>;
    // the register split of the kernel draws on what a block is launched with
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, s2a_fwd_kernel<HD>);
    if (e != cudaSuccess) return e;
    if (a.numRegs < C::kRegsLaunch || a.sharedSizeBytes != 0) return cudaErrorInvalidConfiguration;
    return cudaFuncSetAttribute(s2a_fwd_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
}

}  // namespace

cudaError_t configure_fwd() {
    const cudaError_t e = configure_one<64>();
    return e != cudaSuccess ? e : configure_one<128>();
}

cudaError_t launch_fwd(const FwdParams& p, int d, cudaStream_t stream, bool overlap) {
    const long long n_items = static_cast<long long>(p.geo.B) * p.geo.H * p.geo.groups * p.pairs_per_group;
    const unsigned grid = static_cast<unsigned>(n_items);
    return d == 64 ? launch_kernel(s2a_fwd_kernel<64>, grid, FwdCfg<64>::kThreads, FwdCfg<64>::kSmemBytes, stream, p, overlap)
                   : launch_kernel(s2a_fwd_kernel<128>, grid, FwdCfg<128>::kThreads, FwdCfg<128>::kSmemBytes, stream, p, overlap);
}

}  // namespace s2a
