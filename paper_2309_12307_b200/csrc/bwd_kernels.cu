// S2-Attn backward for sm_100a: the derivative of Algorithm 1 (with Eq. 1 inside each group).
//
// With P = exp(scale * Q K^T - lse) on the attended pairs and D_t = dO_t . o_t:
//     dV = P^T dO          dP = dO V^T          dS = P o (dP - D)
//     dQ = scale * dS K    dK = scale * dS^T Q
// Four kernels:
//   1. preprocess: D[b,h,t] = sum_c dO[b,t,h,c] * o[b,t,h,c]                     (memory bound)
//   2. dQ, recomputing: persistent; a work item is one 128-row query tile, which walks the 128-key tiles of
//            its group (keys <= query) and computes S, dP, dS again
//   3. dK,dV: persistent; a work item is one 128-row key tile, against which the 64-query sub-tiles of
//            every query head that shares the KV head (queries >= key) are streamed, so the sum over
//            those heads stays in tensor memory and needs no atomics.  It works on the transposed
//            scores S^T = K Q^T so that P^T and dS^T come out with keys along tensor-memory lanes, which
//            is the layout the A operand of dV += P^T dO and dK += dS^T Q needs.  Optionally it also
//            leaves dS^T in global memory,
//   4. dQ from spilled dS^T: persistent; a chain of plain products dQ_i = scale * sum_j dS_ij K_j that
//            replaces kernel 2 when the caller's workspace has room for the spill.
// The roll of the shifted heads and the group boundaries are folded into TMA coordinates exactly
// as in the forward kernel; all results are stored at original token rows.
//
// Kernels 2 and 3 share their warp roles (one CTA per SM, all 512 tensor-memory columns):
// warp 0 loads with TMA; warp 1 issues the score MMAs and warp 2 the gradient MMAs (a single issuing
// warp spends so long on its own barrier waits that the tensor pipe runs dry in between; with two, one
// can issue while the other waits); warp 3 owns the tensor-memory allocation (and loads K and V in kernel
// 3); warps 4-11 do the elementwise work with one tensor-memory lane and half of the columns per thread;
// warps 12-15 write finished accumulators out.  S and dP (S^T and dP^T) need one buffer only: the elementwise
// warps copy their part into registers and release it at once, so that the score products of the next
// step run while they work on the current one, and write their bf16 results to columns of their own.
#include "s2a_params.h"
#include "sm100_ptx.cuh"

namespace s2a {

namespace {

constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ int mod_pos(int x, int n) {
    // x in (-n, 2 n)
    if (x < 0) x += n;
    return x >= n ? x - n : x;
}

// ------------------------------------------------------------------------------------------------
// 1. preprocess
// ------------------------------------------------------------------------------------------------
// Bound by the reads of o and dO.  A row of d bf16 values is read by d/8 threads with 16-byte loads, two rows to a
// thread so that four loads are in flight (one row: 9.6 us where two take 7.4; four rows leave fewer
// warps, 24.6 where two take 22.5).  Row numbers are split by multiplication: the three 64-bit divisions that
// stood here kept the issue slots 70 % busy.  32 heads of 128, 8k tokens 26.6 -> 22.5 us, 16k 49.2 -> 41.0, 32k
// 94.7 -> 77.8 (6.9 TB/s); 2 x 4096 tokens of 32 heads of 64 11.2 -> 7.4.
constexpr int kPreRows = 2;
template <int HD>
__global__ void __launch_bounds__(256) s2a_bwd_preprocess_kernel(const PreParams p) {
    constexpr int kThreadsPerRow = HD / 8, kRowsAtOnce = 256 / kThreadsPerRow;
    release_successor();
    wait_for_predecessor();
    const int first = static_cast<int>(blockIdx.x) * (kRowsAtOnce * kPreRows) + static_cast<int>(threadIdx.x) / kThreadsPerRow;
    const int part = threadIdx.x % kThreadsPerRow;
    uint4 a[kPreRows], c[kPreRows];
#pragma unroll
    for (int r = 0; r < kPreRows; ++r) {
        const int row = first + r * kRowsAtOnce;  // (b * N + t) * H + h
        a[r] = c[r] = make_uint4(0, 0, 0, 0);
        if (row < p.rows) {
            a[r] = reinterpret_cast<const uint4*>(p.o + static_cast<long long>(row) * HD)[part];
            c[r] = reinterpret_cast<const uint4*>(p.dO + static_cast<long long>(row) * HD)[part];
        }
    }
#pragma unroll
    for (int r = 0; r < kPreRows; ++r) {
        const uint32_t aw[4] = {a[r].x, a[r].y, a[r].z, a[r].w};
        const uint32_t cw[4] = {c[r].x, c[r].y, c[r].z, c[r].w};
        float acc = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            // a bf16 is the upper half of an fp32
            acc = fmaf(__uint_as_float(aw[e] << 16), __uint_as_float(cw[e] << 16), acc);
            acc = fmaf(__uint_as_float(aw[e] & 0xffff0000u), __uint_as_float(cw[e] & 0xffff0000u), acc);
        }
#pragma unroll
        for (int off = kThreadsPerRow / 2; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        const int row = first + r * kRowsAtOnce;
        if (row < p.rows && part == 0) {
            int h, t;
            const int b = p.by_tokens(p.by_heads(row, &h), &t);
            p.Dsum[(static_cast<long long>(b) * p.H + h) * p.N + t] = acc;
        }
    }
}

// ------------------------------------------------------------------------------------------------
// configuration of the dK,dV kernel, accumulator read-out
// ------------------------------------------------------------------------------------------------
template <int HD>
struct BwdCfg {
    static constexpr int kThreads = 512;  // 4 load and issue warps, 8 elementwise warps, 4 epilogue warps
    static constexpr int kBoxes = HD / 64;
    static constexpr int kBigBoxBytes = kTile * 128;            // 128-row box
    static constexpr int kSubBoxBytes = kSubTile * 128;         // 64-row box
    static constexpr int kBigTileBytes = kBoxes * kBigBoxBytes; // resident operand tile
    static constexpr int kSubTileBytes = kBoxes * kSubBoxBytes; // streamed operand tile
    static constexpr int kStages = 4;
    static constexpr int kStatBytes = kSubTile * 4;             // lse or D of one streamed tile
    static constexpr int kStageBytes = 2 * kSubTileBytes;       // two streamed operands per stage
    static constexpr int kOutBytes = 4 * 2 * 4096;              // two staging buffers for each epilogue warp
    static constexpr int kBarBytes = 1024;
    static constexpr int kNeeded = 2 * kBigTileBytes + kStages * kStageBytes + kOutBytes + kStages * 2 * kStatBytes + kBarBytes;
    // at least 120 KB so that only one CTA fits on an SM: each CTA allocates all of tensor memory
    static constexpr int kSmemBytes = kNeeded > 120 * 1024 ? kNeeded : 120 * 1024;
    static constexpr int kTmemCols = 512;
    // registers per thread after the split; the launch gives kRegsLaunch to each of the 512
    static constexpr int kRegsLaunch = 128, kRegsElem = 152, kRegsOther = 104;
    static_assert(2 * kRegsElem + 2 * kRegsOther <= 4 * kRegsLaunch, "register split");
};

// Store COLS consecutive fp32 accumulator columns of this thread's tensor-memory lane (times `mul`)
// as bf16 to `dst`.
template <int COLS>
__device__ __forceinline__ void store_acc_cols(uint32_t t_addr, float mul, __nv_bfloat16* dst_row, bool row_valid) {
#pragma unroll
    for (int c = 0; c < COLS / 32; ++c) {
        uint32_t r[32];
        tmem_ld_32x32(t_addr + c * 32, r);
        tmem_wait_ld();
        uint4* dst = reinterpret_cast<uint4*>(dst_row + c * 32);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            uint4 pk;
            pk.x = pack_bf16(__uint_as_float(r[8 * e + 0]) * mul, __uint_as_float(r[8 * e + 1]) * mul);
            pk.y = pack_bf16(__uint_as_float(r[8 * e + 2]) * mul, __uint_as_float(r[8 * e + 3]) * mul);
            pk.z = pack_bf16(__uint_as_float(r[8 * e + 4]) * mul, __uint_as_float(r[8 * e + 5]) * mul);
            pk.w = pack_bf16(__uint_as_float(r[8 * e + 6]) * mul, __uint_as_float(r[8 * e + 7]) * mul);
            if (row_valid) dst[e] = pk;
        }
    }
}

// Write 32 accumulator rows of HD columns (times `mul`) as bf16: this warp's tensor-memory lanes at
// `t_addr` go to tokens tok0 .. tok0+31 of `head`, 64 columns at a time through the warp's staging buffers
// (2 x 4 KB of shared memory at `stage`, `used` counts their uses) and a TMA store.  Storing 16 bytes a lane
// straight to rows that lie heads * d apart touches 32 lines with every instruction, 4096 clocks for
// a 128 x 256 tile.  Only the first `valid` rows exist; rows of a ragged tile are stored directly
// (`row_ptr`: this lane's row).  `tm`: box (64, 1, 32, 1).  `done()` runs when the accumulator has been read.
template <int HD, typename Done>
__device__ __forceinline__ void store_acc_rows(const CUtensorMap* tm, uint8_t* stage, uint32_t& used, uint32_t t_addr, float mul,
                                               __nv_bfloat16* row_ptr, int head, int tok0, int b, int valid, Done done) {
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int c = 0; c < HD / 64; ++c) {
        uint32_t r[64];
        tmem_ld_32x32(t_addr + c * 64, *reinterpret_cast<uint32_t(*)[32]>(&r[0]));
        tmem_ld_32x32(t_addr + c * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&r[32]));
        tmem_wait_ld();
        if (c == HD / 64 - 1) done();
        uint8_t* buf = stage + (used & 1) * 4096;
        if (valid >= 32) {
            if (lane == 0) bulk_wait_read<1>();  // the store before the last one has left this buffer
            __syncwarp();
        }
        const uint32_t dst_s = smem_u32(buf) + lane * 128;
        uint4* dst_g = reinterpret_cast<uint4*>(row_ptr + c * 64);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            uint4 pk;
            pk.x = pack_bf16(__uint_as_float(r[8 * e + 0]) * mul, __uint_as_float(r[8 * e + 1]) * mul);
            pk.y = pack_bf16(__uint_as_float(r[8 * e + 2]) * mul, __uint_as_float(r[8 * e + 3]) * mul);
            pk.z = pack_bf16(__uint_as_float(r[8 * e + 4]) * mul, __uint_as_float(r[8 * e + 5]) * mul);
            pk.w = pack_bf16(__uint_as_float(r[8 * e + 6]) * mul, __uint_as_float(r[8 * e + 7]) * mul);
            if (valid >= 32) {
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst_s + ((e ^ (lane & 7)) << 4)), "r"(pk.x), "r"(pk.y),
                             "r"(pk.z), "r"(pk.w)
                             : "memory");
            } else if (lane < valid) {
                dst_g[e] = pk;
            }
        }
        if (valid >= 32) {
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
                tma_store_4d(tm, buf, c * 64, head, tok0, b);
                bulk_commit_group();
            }
            ++used;
        }
    }
}

// ------------------------------------------------------------------------------------------------
// 2. dQ
// ------------------------------------------------------------------------------------------------
// A work item is a 128-row query tile; it walks the 128-key tiles j_begin..i of its group (keys <= query).
// Per key tile n:  S_n = Q K_n^T,  dP_n = dO V_n^T,  dS_n = P_n o (dP_n - D) as bf16,
// dQ += dS_n K_n  (K_n is MN-major in the tile that served Q K_n^T).
// Full 128x128 score products: a 64-column product re-reads the 128-row A operand from shared memory
// for half the work and runs at 48 instead of 32 clocks per K step.
//
// Tensor memory columns: dQ [0,HD)   S [128,256)   dP [256,384)   dS (bf16, two buffers) [384,448) [448,512)
// The elementwise warps copy S and dP into registers at the start of a step and release them at once, so the
// score products of the next step run while they work.  Shared memory: Q and dO of the item resident, a ring
// of three K tiles and a ring of two V tiles.
//
// Persistent, like the dK,dV kernel: items by cluster launch control, the loads of the next item behind those
// of the last one, the accumulator read out by four warps of their own beside the next item's first steps.
// Before (a block for each tile, dS over S, dP copied ahead) and after, us a launch in a loop: Llama2-7B 8k 246 and
// 202, 16k 808 and 677, 32k 2720 and 2580 (at the power limit), 4 x 2000 tokens with groups of 200 48 and 27,
// grouped query 2 x 4096 125 and 84.
template <int HD>
struct DqCfg {
    static constexpr int kThreads = 512;  // 4 load and issue warps, 8 elementwise warps, 4 epilogue warps
    static constexpr int kBoxes = HD / 64;
    static constexpr int kBoxBytes = kTile * 128;          // 128 rows x 128 bytes
    static constexpr int kTileBytes = kBoxes * kBoxBytes;  // one Q, dO, K or V tile
    // K_n serves S_n early in step n-1 and the dQ MMAs at the end of step n: three K tiles are live
    // around the issue of S_{n+1}, V_n only until dP_n is done.
    static constexpr int kRingK = 3;
    static constexpr int kRingV = 2;
    static constexpr int kBarBytes = 1024;
    static constexpr int kNeeded = (2 + kRingK + kRingV) * kTileBytes + kBarBytes;
    // at least 120 KB so that only one CTA fits on an SM: each CTA allocates all of tensor memory
    static constexpr int kSmemBytes = kNeeded > 120 * 1024 ? kNeeded : 120 * 1024;
    static constexpr int kTmemCols = 512;
    // registers per thread after the split; the launch gives kRegsLaunch to each of the 512
    static constexpr int kRegsLaunch = 128, kRegsElem = 168, kRegsOther = 88;
    static_assert(2 * kRegsElem + 2 * kRegsOther <= 4 * kRegsLaunch, "register split");
};

struct DqItem {
    int b, h, hk;     // b = -1: no more items
    int tq0, q_valid; // the query tile
    int j_begin, n_steps;
    GroupLayout L;
};
// Work item `id` (heaviest query tiles of a chunk of units first); false marks a slot of a group that has
// fewer tiles than the largest one.
__device__ __forceinline__ bool dq_item(const BwdDqParams& p, int id, DqItem* t) {
    const Geometry& geo = p.geo;
    int unit, rank, g;
    p.order.decode(id, &unit, &rank);
    t->b = p.by_heads(geo.by_groups(unit, &g), &t->h);
    t->hk = geo.by_rep(t->h);
    t->L = group_layout(geo, (t->h < geo.n_unshifted) ? 0 : geo.shift, g);
    const int i = t->L.nTiles - 1 - rank;
    if (i < 0) return false;
    t->j_begin = first_key_tile(t->L, i);
    t->n_steps = i + 1 - t->j_begin;
    const TileRef tq = tile_ref(t->L, i);
    t->tq0 = tq.tok0, t->q_valid = tq.valid;
    return true;
}

struct DqBars {
    uint64_t res_full, res_empty;    // Q and dO of an item landed / the score products of the item are done
    uint64_t acc_full, acc_empty;    // dQ of an item is complete / has been read out
    uint64_t drain, drain2;          // abort path only (gradient / score MMA warp)
    uint64_t s_full;                 // S_n and dP_n are in tensor memory
    uint64_t s_free;                 // the elementwise threads hold them in registers
    uint64_t p_full[2], p_free[2];   // bf16 dS_n is in tensor memory / the dQ MMAs that read it are done
    uint64_t k_full[3], k_empty[3], v_full[2], v_empty[2];
    uint64_t sched_full[8];
    uint64_t clc;
    alignas(16) uint8_t clc_resp[16];
    DqItem item[8];
    uint32_t tmem_slot;
    int abort_flag;
};
static_assert(sizeof(DqBars) <= 1024, "barrier block");

template <int HD>
__global__ void __launch_bounds__(DqCfg<HD>::kThreads, 1) s2a_bwd_dq_kernel(const __grid_constant__ BwdDqParams p) {
    using C = DqCfg<HD>;
    constexpr int kSched = 8;  // items in flight
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = smem_raw;                          // 1024-byte aligned: nothing precedes the dynamic array
    uint8_t* sQ = smem;                                // resident: Q_i
    uint8_t* sDO = sQ + C::kTileBytes;                 // resident: dO_i
    uint8_t* sK = sDO + C::kTileBytes;                 // ring of K tiles
    uint8_t* sV = sK + C::kRingK * C::kTileBytes;      // ring of V tiles
    DqBars* bars = reinterpret_cast<DqBars*>(sV + C::kRingV * C::kTileBytes);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const Geometry& geo = p.geo;

    if (threadIdx.x == 0) {
        // hand-offs by whole warps count one arrival per warp
        mbar_init(&bars->res_full, 1);
        mbar_init(&bars->res_empty, 1);
        mbar_init(&bars->acc_full, 1);
        mbar_init(&bars->acc_empty, 4);
        mbar_init(&bars->drain, 1);
        mbar_init(&bars->drain2, 1);
        mbar_init(&bars->s_full, 1);
        mbar_init(&bars->s_free, 8);
        for (int x = 0; x < 2; ++x) {
            mbar_init(&bars->p_full[x], 8);
            mbar_init(&bars->p_free[x], 1);
            mbar_init(&bars->v_full[x], 1);
            mbar_init(&bars->v_empty[x], 1);
        }
        for (int x = 0; x < C::kRingK; ++x) {
            mbar_init(&bars->k_full[x], 1);
            mbar_init(&bars->k_empty[x], 1);
        }
        for (int x = 0; x < kSched; ++x) mbar_init(&bars->sched_full[x], 1);
        mbar_init(&bars->clc, 1);
        fence_barrier_init();
        tma_prefetch_desc(&p.tm_q);
        tma_prefetch_desc(&p.tm_do);
        tma_prefetch_desc(&p.tm_k);
        tma_prefetch_desc(&p.tm_v);
    }
    if (warp == 3) {
        tmem_alloc(&bars->tmem_slot, C::kTmemCols);
        tmem_relinquish();
    }
    wait_for_predecessor();
    // A bounded wait that expired earlier (in any kernel) leaves the status word set: later CTAs
    // then return at once instead of each running into its own time limit.
    if (threadIdx.x == 0) bars->abort_flag = *reinterpret_cast<volatile int*>(p.status);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    release_successor();
    const uint32_t tmem_base = bars->tmem_slot;
    if (bars->abort_flag != 0) {
        if (warp == 3) tmem_dealloc(tmem_base, C::kTmemCols);
        return;
    }
    const WaitCtx ctx{&bars->abort_flag, p.status, p.host_status};
    constexpr uint32_t kColAcc = 0, kColS = 128, kColP = 256, kColDs = 384;

    // Every consumer warp walks the same sequence of items: the k-th one, false = the end (or aborting).
    auto next_item = [&](int k, int where, DqItem* t) -> bool {
        if (!mbar_wait_uniform(&bars->sched_full[k % kSched], (k / kSched) & 1, ctx, where)) return false;
        *t = bars->item[k % kSched];
        return t->b >= 0;
    };

    if (warp < 4) {
        setmaxnreg_dec<C::kRegsOther>();
        if (warp == 0) {
            // ---- work items and TMA loads
            if (lane == 0) {
                int it = 0;     // key tiles requested so far
                int n_res = 0;  // items whose Q and dO were requested
                bool ok = true;
                ItemSource items{&bars->clc, bars->clc_resp};
                int id = static_cast<int>(blockIdx.x);
                for (int k = 0; ok; ++k) {
                    DqItem t;
                    while (id >= 0 && !dq_item(p, id, &t)) id = items.next(ctx, kWaitBwdDq + 12, &ok);
                    if (id < 0) t.b = -1;
                    bars->item[k % kSched] = t;
                    mbar_arrive(&bars->sched_full[k % kSched]);  // release: the item is visible to whoever sees the phase
                    if (id < 0) break;
                    for (int n = 0; ok && n < t.n_steps; ++n, ++it) {
                        const int st = it % C::kRingV, sk = it % C::kRingK;
                        const int tk0 = tile_ref(t.L, t.j_begin + n).tok0;
                        if (!mbar_wait(&bars->v_empty[st], ((it / C::kRingV) & 1) ^ 1, ctx, kWaitBwdDq + 1)) { ok = false; break; }
                        mbar_expect_tx(&bars->v_full[st], C::kTileBytes);
                        for (int bx = 0; bx < C::kBoxes; ++bx)
                            tma_load_4d(sV + st * C::kTileBytes + bx * C::kBoxBytes, &p.tm_v, &bars->v_full[st], bx * 64, t.hk, tk0, t.b);
                        if (n == 0) {
                            if (!mbar_wait(&bars->res_empty, (k & 1) ^ 1, ctx, kWaitBwdDq + 13)) {
                                mbar_wait_drain(&bars->v_full[st], (it / C::kRingV) & 1);
                                ok = false;
                                break;
                            }
                            mbar_expect_tx(&bars->res_full, 2 * C::kTileBytes);
                            for (int bx = 0; bx < C::kBoxes; ++bx) {
                                tma_load_4d(sQ + bx * C::kBoxBytes, &p.tm_q, &bars->res_full, bx * 64, t.h, t.tq0, t.b);
                                tma_load_4d(sDO + bx * C::kBoxBytes, &p.tm_do, &bars->res_full, bx * 64, t.h, t.tq0, t.b);
                            }
                            ++n_res;
                        }
                        if (!mbar_wait(&bars->k_empty[sk], ((it / C::kRingK) & 1) ^ 1, ctx, kWaitBwdDq + 8)) {
                            mbar_wait_drain(&bars->v_full[st], (it / C::kRingV) & 1);
                            ok = false;
                            break;
                        }
                        mbar_expect_tx(&bars->k_full[sk], C::kTileBytes);
                        for (int bx = 0; bx < C::kBoxes; ++bx)
                            tma_load_4d(sK + sk * C::kTileBytes + bx * C::kBoxBytes, &p.tm_k, &bars->k_full[sk], bx * 64, t.hk, tk0, t.b);
                    }
                    if (ok) id = items.next(ctx, kWaitBwdDq + 12, &ok);
                }
                if (bars->abort_flag != 0) {
                    // let loads that are still in flight land before the CTA gives its memory back
                    if (n_res > 0) mbar_wait_drain(&bars->res_full, (n_res - 1) & 1);
                    for (int nn = (it > C::kRingK ? it - C::kRingK : 0); nn < it; ++nn)
                        mbar_wait_drain(&bars->k_full[nn % C::kRingK], (nn / C::kRingK) & 1);
                    for (int nn = (it > C::kRingV ? it - C::kRingV : 0); nn < it; ++nn)
                        mbar_wait_drain(&bars->v_full[nn % C::kRingV], (nn / C::kRingV) & 1);
                }
            }
            __syncwarp();
        } else if (warp == 1) {
            // ---- score MMAs: dP_n = dO V_n^T and S_n = Q K_n^T, as soon as the elementwise warps hold those of the
            // step before in registers.  The whole warp walks the loop so that addresses and descriptors
            // stay warp-uniform values; only the MMA and commit instructions are issued by one elected lane.
            constexpr uint32_t idesc_sc = idesc_bf16(128, kTile, 0, 0);
            const uint32_t dQ = desc_lo_k_major(smem_u32(sQ)), dDO = desc_lo_k_major(smem_u32(sDO));
            const uint32_t tP = tmem_base + kColP, tS = tmem_base + kColS;
            int it = 0;
            bool ok = true;
            for (int k = 0; ok; ++k) {
                DqItem t;
                if (!next_item(k, kWaitBwdDq + 14, &t)) break;
                if (!mbar_wait_uniform(&bars->res_full, k & 1, ctx, kWaitBwdDq + 3)) break;
                for (int n = 0; n < t.n_steps; ++n, ++it) {
                    const int st = it % C::kRingV, sk = it % C::kRingK;
                    // the two TMA barriers first: they have usually completed long ago
                    if (!mbar_wait_uniform(&bars->v_full[st], (it / C::kRingV) & 1, ctx, kWaitBwdDq + 2) ||
                        !mbar_wait_uniform(&bars->k_full[sk], (it / C::kRingK) & 1, ctx, kWaitBwdDq + 10)) { ok = false; break; }
                    if (it >= 1 && !mbar_wait_uniform(&bars->s_free, (it - 1) & 1, ctx, kWaitBwdDq + 9)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t dV = desc_lo_k_major(smem_u32(sV + st * C::kTileBytes));
                    const uint32_t dK = desc_lo_k_major(smem_u32(sK + sk * C::kTileBytes));
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < HD / 16; ++kk)
                            mma_ss(tP, dDO + desc_step_k_major(kk, C::kBoxBytes), dV + desc_step_k_major(kk, C::kBoxBytes), idesc_sc, kk > 0);
                        mma_commit(&bars->v_empty[st]);
#pragma unroll
                        for (int kk = 0; kk < HD / 16; ++kk)
                            mma_ss(tS, dQ + desc_step_k_major(kk, C::kBoxBytes), dK + desc_step_k_major(kk, C::kBoxBytes), idesc_sc, kk > 0);
                        mma_commit(&bars->s_full);
                        if (n == t.n_steps - 1) mma_commit(&bars->res_empty);
                    }
                    __syncwarp();
                }
            }
            if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&bars->abort_flag) != 0)) {
                if (elect_one()) {
                    mma_commit(&bars->drain2);
                    mbar_wait_drain(&bars->drain2, 0);
                }
            }
            __syncwarp();
        } else if (warp == 2) {
            // ---- gradient MMAs: dQ += dS_n K_n
            constexpr uint32_t idesc_acc = idesc_bf16(128, HD, 0, 1);
            int it = 0;
            bool ok = true;
            for (int k = 0; ok; ++k) {
                DqItem t;
                if (!next_item(k, kWaitBwdDq + 15, &t)) break;
                // the first product of an item overwrites the accumulator: the previous item's must have been read out
                if (k > 0 && !mbar_wait_uniform(&bars->acc_empty, (k - 1) & 1, ctx, kWaitBwdDq + 7)) break;
                for (int n = 0; n < t.n_steps; ++n, ++it) {
                    const int bf = it & 1, sk = it % C::kRingK;
                    if (!mbar_wait_uniform(&bars->p_full[bf], (it >> 1) & 1, ctx, kWaitBwdDq + 4)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t dKmn = desc_lo_mn_major(smem_u32(sK + sk * C::kTileBytes), C::kBoxBytes);
                    const uint32_t tdS = tmem_base + kColDs + bf * 64;
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < kTile / 16; ++kk)
                            mma_ts(tmem_base + kColAcc, tdS + kk * 8, dKmn + kk * kDescStepMn, idesc_acc, (n > 0) || (kk > 0));
                        mma_commit(&bars->k_empty[sk]);
                        mma_commit(&bars->p_free[bf]);
                        if (n == t.n_steps - 1) mma_commit(&bars->acc_full);
                    }
                    __syncwarp();
                }
            }
            if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&bars->abort_flag) != 0)) {
                // MMAs already issued must finish before tensor memory is released
                if (elect_one()) {
                    mma_commit(&bars->drain);
                    mbar_wait_drain(&bars->drain, 0);
                }
            }
            __syncwarp();
        }
        // warp 3: owns the tensor-memory allocation only
    } else if (warp < 12) {
        // ---- elementwise: thread (quad, lane, half) owns columns [64 half, +64) of score row 32 quad + lane
        setmaxnreg_inc<C::kRegsElem>();
        const int quad = warp & 3;
        const int half = (warp - 4) >> 2;
        const int row = quad * 32 + lane;
        const uint32_t t_row = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
        const float c2 = p.scale_log2;
        const uint64_t c2x2 = f2_pack(c2, c2);
        int it = 0;
        bool ok = true;
        for (int k = 0; ok; ++k) {
            DqItem t;
            if (!next_item(k, kWaitBwdDq + 16, &t)) break;
            // rows past the end of a ragged tile are not part of the group: they are computed on whatever
            // the box holds there and never stored
            const bool row_valid = row < t.q_valid;
            const size_t stat_idx = (static_cast<size_t>(t.b) * geo.H + t.h) * geo.N + t.tq0 + row;
            const float neg_lse2 = row_valid ? -p.lse[stat_idx] * kLog2e : 0.f;
            const float Drow = row_valid ? p.Dsum[stat_idx] : 0.f;
            const uint64_t nlx2 = f2_pack(neg_lse2, neg_lse2), Dx2 = f2_pack(Drow, Drow);
            for (int n = 0; n < t.n_steps; ++n, ++it) {
                const int bf = it & 1;
                // Key x of the tile is visible to query row r iff it is one of the tile's valid rows and,
                // in the diagonal tile, x <= r.  Off the diagonal a full tile needs no mask at all.
                const int k_valid = tile_ref(t.L, t.j_begin + n).valid;
                if (!mbar_wait_uniform(&bars->s_full, it & 1, ctx, kWaitBwdDq + 11)) { ok = false; break; }
                tc_fence_after();
                uint32_t sr[2][32], dp[2][32];
                tmem_ld_32x32(t_row + kColS + half * 64, sr[0]);
                tmem_ld_32x32(t_row + kColS + half * 64 + 32, sr[1]);
                tmem_ld_32x32(t_row + kColP + half * 64, dp[0]);
                tmem_ld_32x32(t_row + kColP + half * 64 + 32, dp[1]);
                tmem_wait_ld();
                tc_fence_before();
                mbar_arrive_warp(&bars->s_free);
                if (it >= 2 && !mbar_wait_uniform(&bars->p_free[bf], ((it >> 1) & 1) ^ 1, ctx, kWaitBwdDq + 5)) { ok = false; break; }
                tc_fence_after();
                const bool last = (n == t.n_steps - 1);
                const bool masked = last || k_valid < kTile;
                const int vis = (last && row < k_valid) ? row : k_valid - 1;
                const int lim = vis - half * 64;  // visible iff (column within this half) <= lim
                const uint32_t tdS = t_row + kColDs + bf * 64 + half * 32;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t pk[16];
                    if (masked) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            float pe0 = fast_exp2(fmaf(__uint_as_float(sr[c][2 * e]), c2, neg_lse2));
                            float pe1 = fast_exp2(fmaf(__uint_as_float(sr[c][2 * e + 1]), c2, neg_lse2));
                            if (c * 32 + 2 * e > lim) pe0 = 0.f;
                            if (c * 32 + 2 * e + 1 > lim) pe1 = 0.f;
                            pk[e] = pack_bf16(pe0 * (__uint_as_float(dp[c][2 * e]) - Drow), pe1 * (__uint_as_float(dp[c][2 * e + 1]) - Drow));
                        }
                    } else {
                        // two columns per instruction for the multiply-adds
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            const uint64_t x = f2_fma(f2_pack(__uint_as_float(sr[c][2 * e]), __uint_as_float(sr[c][2 * e + 1])), c2x2, nlx2);
                            float x0, x1;
                            f2_unpack(x, x0, x1);
                            // part of the exponentials goes to the FMA pipe (see poly_exp2_x2)
                            const uint64_t pe = ((kPolyExpMask >> e) & 1u) ? poly_exp2_x2(x) : f2_pack(fast_exp2(x0), fast_exp2(x1));
                            const uint64_t u = f2_sub(f2_pack(__uint_as_float(dp[c][2 * e]), __uint_as_float(dp[c][2 * e + 1])), Dx2);
                            float d0, d1;
                            f2_unpack(f2_mul(pe, u), d0, d1);
                            pk[e] = pack_bf16(d0, d1);
                        }
                    }
                    tmem_st_32x16(tdS + c * 16, pk);
                }
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive_warp(&bars->p_full[bf]);
            }
        }
    } else {
        // ---- epilogue: thread owns accumulator row 32 quad + lane
        setmaxnreg_dec<C::kRegsOther>();
        const int quad = warp & 3;
        const int row = quad * 32 + lane;
        const uint32_t t_row = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
        for (int k = 0;; ++k) {
            DqItem t;
            if (!next_item(k, kWaitBwdDq + 17, &t)) break;
            if (!mbar_wait_uniform(&bars->acc_full, k & 1, ctx, kWaitBwdDq + 6)) break;
            tc_fence_after();
            __nv_bfloat16* dst = p.dq + (static_cast<size_t>(t.b) * geo.N + t.tq0 + row) * p.dq_tok_stride + static_cast<size_t>(t.h) * HD;
            store_acc_cols<HD>(t_row + kColAcc, p.scale, dst, row < t.q_valid);
            tc_fence_before();
            mbar_arrive_warp(&bars->acc_empty);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 3) {
        tc_fence_after();
        tmem_dealloc(tmem_base, C::kTmemCols);
    }
}

// ------------------------------------------------------------------------------------------------
// 3. dK, dV
// ------------------------------------------------------------------------------------------------
// Tensor memory columns: dV, dK (HD each), S^T, dP^T (64 each), P^T and dS^T (bf16, 64 together; two buffers where
//                        HD = 64 leaves room), K (bf16, HD/2: the A operand of S^T = K Q^T), where HD = 64 V likewise
//                        (the A operand of dP^T = V dO^T: the products read less shared memory, and V of the next item
//                        comes as early as its K; 2 x 4096 tokens grouped query 166,000 -> 161,000 clocks a launch,
//                        32k 3,838,000 -> 3,657,000)
// One buffer of S^T and dP^T is enough: the elementwise warps copy them into registers at the start of a step
// and release them at once, so the score products of the next step run while they work.  P^T and dS^T are
// written when the gradient MMAs are done with what the buffer held.  With P^T and dS^T over S^T, in two
// buffers, the score products waited some 400 clocks a step for the gradient MMAs.  Microseconds a launch in a
// loop, before and after (plain / spilling): Llama2-7B 32k 3670 and 3475 / 4270 and 4150, 16k 992 and 943 / 1149 and
// 1094, 8k 281 and 275 / 328 and 313; head size 64 at 32k 2557 and 2503 / 3151 and 3053.
//
// The CTA owns key tile (b, hk, original tokens tk0 .. tk0+127).  For every query head hq that
// reads KV head hk (shift s): the tile sits at rolled position (tk0 - s) mod N, i.e. in group g at
// key tile j, and is attended by query sub-tiles (64 rows) 2j .. 2*nTiles-1 of that group.  (When the
// tiles are ragged the host only admits KV heads whose query heads all have the same shift, so the
// key tile is a tile of every head's partition.)
struct HeadWalk {
    GroupLayout L;
    int g, j, n_begin, n_end;
};
__device__ __forceinline__ HeadWalk head_walk(const Geometry& geo, int hq, int tk0) {
    HeadWalk w;
    const int s = (hq < geo.n_unshifted) ? 0 : geo.shift;
    const int pos = mod_pos(tk0 - s, geo.N);
    int in_group;
    w.g = geo.by_group(pos, &in_group);
    w.L = group_layout(geo, s, w.g);
    const int nB = w.L.nTiles - w.L.nA;
    w.j = in_group < w.L.lenA ? (w.L.swapped ? nB : 0) + in_group / kTile
                              : (w.L.swapped ? 0 : w.L.nA) + (in_group - w.L.lenA) / kTile;
    w.n_begin = 2 * w.j;
    w.n_end = 2 * end_query_tile(w.L, w.j);
    return w;
}

// A work item of the dK,dV kernel: key tile `j0` (in the partition of the KV head's first query head) of
// unit (b, hk, g0), in the block order shared by all kernels.  total_steps = 0 marks a slot of a group
// that has fewer tiles than the largest one.
struct DkDvItem {
    int b, hk, tk0, k_valid, total_steps;
};
__device__ __forceinline__ DkDvItem dkdv_item(const BwdDkDvParams& p, long long id) {
    const Geometry& geo = p.geo;
    const SpillPass& pass = p.pass;
    DkDvItem t;
    int unit, j0, g0;
    p.order.decode(static_cast<int>(id), &unit, &j0);
    const int rep = geo.rep;
    t.b = p.by_heads(geo.by_groups(unit, &g0), &t.hk);
    t.hk += pass.hk0;
    const int hq0 = t.hk * rep;
    const int s0 = (hq0 < geo.n_unshifted) ? 0 : geo.shift;
    const GroupLayout L0 = group_layout(geo, s0, g0);
    t.total_steps = 0;
    t.tk0 = 0, t.k_valid = 0;
    if (j0 >= L0.nTiles) return t;
    const TileRef tk = tile_ref(L0, j0);
    t.tk0 = tk.tok0;
    t.k_valid = tk.valid;
    for (int hq = hq0; hq < hq0 + rep; ++hq) {
        const HeadWalk w = head_walk(geo, hq, t.tk0);
        t.total_steps += w.n_end - w.n_begin;
    }
    return t;
}

// Barriers of the dK,dV kernel.  Steps are counted through all items of the CTA (`it`), so the rings of
// stages and score buffers simply carry on from one item to the next.
template <int kStages>
struct DkDvBars {
    uint64_t k_full, v_full;      // K / V of an item landed (one phase per item)
    uint64_t kt_full;             // K (HD = 64: and V) of an item has been copied into tensor memory
    uint64_t v_empty;             // HD = 128: the dP^T products of an item are done, V may be overwritten
    uint64_t s_done;              // all score products of an item are done: the copies may be overwritten
    uint64_t acc_full;            // all gradient MMAs of an item are done
    uint64_t acc_empty;           // the accumulators of an item have been read out
    uint64_t drain;               // abort path only (gradient MMA warp)
    uint64_t drain2;              // abort path only (score MMA warp)
    uint64_t s_full;              // S^T and dP^T of a step are in tensor memory
    uint64_t s_free;              // the elementwise threads of a step hold their S^T and dP^T in registers
    uint64_t p_full[2];           // bf16 P^T and dS^T of a step are in tensor memory (buffer it % kPBufs)
    uint64_t p_free[2];           // the gradient MMAs that read them are done
    uint64_t st_full[kStages];    // streamed operands of a stage landed
    uint64_t st_empty[kStages];   // MMAs reading a stage are done
    uint64_t sched_full[8];       // a work item has been published
    uint64_t clc;
    alignas(16) uint8_t clc_resp[16];
    DkDvItem item[8];             // total_steps = 0: no more items
    uint32_t tmem_slot;
    int abort_flag;
};

// kSpill: every step's dS^T also goes to global memory (see SpillPass) for s2a_bwd_dq_spill_kernel.
//
// Persistent: one CTA per SM takes over key tiles, heaviest first, by cluster launch control.  Everything
// that belongs to the change from one item to the next runs beside the steps: the ids and the streamed
// tiles are requested ahead (warp 0); K of the next item is loaded as soon as the current one has been
// copied to tensor memory, V likewise where it is copied as well (HD = 64), else as soon as the last dP^T
// product is done (warp 3); the copies and the read-out of the accumulators have four warps of their own, so that the elementwise warps go straight on
// with the next item's first steps.  With the elementwise warps doing it and every warp decoding the item
// for itself (64-bit divisions, one after the other), the change of item cost 10,000 to 17,000 clocks, as
// much as ten steps.  Before and after, spilling form, us a launch in a loop: Llama2-7B 8k 354 and 325, 4 x 2048
// tokens with groups of 512 178 and 146, 4 x 2000 with groups of 200 (head size 64) 53 and 43, 32k 4380 and 4290
// (there the part is at its power limit).
template <int HD, bool kSpill>
__global__ void __launch_bounds__(BwdCfg<HD>::kThreads, 1) s2a_bwd_dkdv_kernel(const __grid_constant__ BwdDkDvParams p) {
    using C = BwdCfg<HD>;
    using Bars = DkDvBars<C::kStages>;
    constexpr int kPBufs = HD == 64 ? 2 : 1;  // buffers of P^T and dS^T
    constexpr bool kVInTmem = HD == 64;       // V is a tensor-memory operand like K
    constexpr int kCols = 32;  // query columns per elementwise thread and step: two threads share a key row
    constexpr int kChunks = kCols / 16;
    constexpr int kSched = 8;  // item ids in flight: the TMA warp is at most five items ahead of the read-out
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = smem_raw;                          // 1024-byte aligned: nothing precedes the dynamic array
    uint8_t* sK = smem;                                // resident: K_j
    uint8_t* sV = sK + C::kBigTileBytes;               // resident: V_j
    uint8_t* sStage = sV + C::kBigTileBytes;           // per stage: Q_n then dO_n
    uint8_t* sOut = sStage + C::kStages * C::kStageBytes;  // staging buffers of the epilogue warps
    float* sStat = reinterpret_cast<float*>(sOut + C::kOutBytes);  // per stage: lse[64], D[64]
    Bars* bars = reinterpret_cast<Bars*>(reinterpret_cast<uint8_t*>(sStat) + C::kStages * 2 * C::kStatBytes);
    static_assert(sizeof(Bars) <= C::kBarBytes, "barrier block");

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    // A bounded wait that expired earlier (in any kernel) leaves the status word set: later CTAs
    // then return at once instead of each running into its own time limit.
    if (threadIdx.x == 0) bars->abort_flag = *reinterpret_cast<volatile int*>(p.status);
    __syncthreads();
    if (bars->abort_flag != 0) return;
    __syncthreads();
    const Geometry& geo = p.geo;
    const int rep = geo.rep;
    const int Tg = geo.tiles_per_group;

    if (threadIdx.x == 0) {
        // hand-offs by whole warps count one arrival per warp
        mbar_init(&bars->k_full, 1);
        mbar_init(&bars->v_full, 1);
        mbar_init(&bars->kt_full, 4);
        mbar_init(&bars->v_empty, 1);
        mbar_init(&bars->s_done, 1);
        mbar_init(&bars->acc_full, 1);
        mbar_init(&bars->acc_empty, 4);
        mbar_init(&bars->drain, 1);
        mbar_init(&bars->drain2, 1);
        mbar_init(&bars->s_full, 2);  // the score MMAs are done; their issuer has seen the stage land
        mbar_init(&bars->s_free, 8);
        for (int x = 0; x < kPBufs; ++x) {
            mbar_init(&bars->p_full[x], 8);
            mbar_init(&bars->p_free[x], 1);
        }
        for (int st = 0; st < C::kStages; ++st) {
            mbar_init(&bars->st_full[st], 1);
            mbar_init(&bars->st_empty[st], 1);
        }
        for (int x = 0; x < kSched; ++x) mbar_init(&bars->sched_full[x], 1);
        mbar_init(&bars->clc, 1);
        bars->abort_flag = 0;
        fence_barrier_init();
        tma_prefetch_desc(&p.tm_q);
        tma_prefetch_desc(&p.tm_do);
        tma_prefetch_desc(&p.tm_k);
        tma_prefetch_desc(&p.tm_v);
        tma_prefetch_desc(&p.tm_dk);
        tma_prefetch_desc(&p.tm_dv);
    }
    if (warp == 3) {
        tmem_alloc(&bars->tmem_slot, C::kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = bars->tmem_slot;
    const WaitCtx ctx{&bars->abort_flag, p.status, p.host_status};
    constexpr uint32_t kColDV = 0, kColDK = HD, kColS = 2 * HD, kColP = kColS + 64, kColPdS = kColP + 64, kColKt = kColPdS + 64 * kPBufs,
                       kColVt = kColKt + HD / 2;
    static_assert(kColVt + (kVInTmem ? HD / 2 : 0) <= C::kTmemCols, "tensor memory");

    // Every consumer warp walks the same sequence of items, as the scheduling thread has decoded them (the
    // divisions cost a warp more than a step): the k-th one, false = the end (or aborting).
    auto next_item = [&](int k, int where, DkDvItem* t) -> bool {
        if (!mbar_wait_uniform(&bars->sched_full[k % kSched], (k / kSched) & 1, ctx, where)) return false;
        *t = bars->item[k % kSched];
        return t->total_steps > 0;
    };

    if (warp < 4) {
        setmaxnreg_dec<C::kRegsOther>();
        if (warp == 0) {
            // ---- work items and streamed query sub-tiles
            if (lane == 0) {
                int it = 0;
                bool ok = true;
                ItemSource items{&bars->clc, bars->clc_resp};
                int id = static_cast<int>(blockIdx.x);
                for (int k = 0; ok; ++k) {
                    // the next item that has work; the other warps only see real items and the end marker
                    DkDvItem t;
                    while (id >= 0 && (t = dkdv_item(p, id)).total_steps == 0) {
                        id = items.next(ctx, kWaitBwdDkDv + 10, &ok);
                    }
                    if (id < 0) t.total_steps = 0;
                    bars->item[k % kSched] = t;
                    mbar_arrive(&bars->sched_full[k % kSched]);  // release: the item is visible to whoever sees the phase
                    if (id < 0) break;
                    const int hq0 = t.hk * rep;
                    for (int hq = hq0; ok && hq < hq0 + rep; ++hq) {
                        const HeadWalk w = head_walk(geo, hq, t.tk0);
                        for (int n = w.n_begin; n < w.n_end; ++n, ++it) {
                            const int st = it % C::kStages;
                            const uint32_t ph = (it / C::kStages) & 1;
                            const TileRef tq = subtile_ref(w.L, n);
                            const int tq0 = tq.tok0;
                            // statistics of the valid rows only (a multiple of 4 rows, so of 16 bytes): a ragged
                            // sub-tile must not read past the end of the arrays
                            const uint32_t stat_bytes = static_cast<uint32_t>(tq.valid) * 4u;
                            if (!mbar_wait(&bars->st_empty[st], ph ^ 1, ctx, kWaitBwdDkDv + 1)) { ok = false; break; }
                            mbar_expect_tx(&bars->st_full[st], C::kStageBytes + 2 * stat_bytes);
                            uint8_t* sQ = sStage + st * C::kStageBytes;
                            uint8_t* sDO = sQ + C::kSubTileBytes;
                            for (int bx = 0; bx < C::kBoxes; ++bx) {
                                tma_load_4d(sQ + bx * C::kSubBoxBytes, &p.tm_q, &bars->st_full[st], bx * 64, hq, tq0, t.b);
                                tma_load_4d(sDO + bx * C::kSubBoxBytes, &p.tm_do, &bars->st_full[st], bx * 64, hq, tq0, t.b);
                            }
                            const size_t stat_idx = (static_cast<size_t>(t.b) * geo.H + hq) * geo.N + tq0;
                            if (stat_bytes != 0) {
                                bulk_load_1d(sStat + st * 2 * kSubTile, p.lse + stat_idx, stat_bytes, &bars->st_full[st]);
                                bulk_load_1d(sStat + st * 2 * kSubTile + kSubTile, p.Dsum + stat_idx, stat_bytes, &bars->st_full[st]);
                            }
                        }
                    }
                    if (ok) id = items.next(ctx, kWaitBwdDkDv + 10, &ok);
                }
                if (bars->abort_flag != 0) {
                    // let loads that are still in flight land before the CTA gives its memory back
                    for (int nn = (it > C::kStages ? it - C::kStages : 0); nn < it; ++nn)
                        mbar_wait_drain(&bars->st_full[nn % C::kStages], (nn / C::kStages) & 1);
                }
            }
            __syncwarp();
        } else if (warp == 1) {
            // ---- score MMAs of step `it`: dP^T = V dO^T and S^T = K Q^T, as soon as the elementwise warps hold those
            // of the step before in registers (warp-uniform loop, one elected lane issues; see the dQ kernel)
            constexpr uint32_t idesc_sc = idesc_bf16(128, kSubTile, 0, 0);
            const uint32_t dV = desc_lo_k_major(smem_u32(sV));
            const uint32_t tP = tmem_base + kColP, tKt = tmem_base + kColKt, tVt = tmem_base + kColVt;
            int it = 0;
            bool ok = true;
            for (int k = 0; ok; ++k) {
                DkDvItem t;
                if (!next_item(k, kWaitBwdDkDv + 11, &t)) break;
                const int steps = t.total_steps;
                if (!mbar_wait_uniform(&bars->kt_full, k & 1, ctx, kWaitBwdDkDv + 16)) break;
                for (int x = 0; ok && x < steps; ++x, ++it) {
                    const int st = it % C::kStages;
                    const bool last = x == steps - 1;
                    if (!mbar_wait_uniform(&bars->st_full[st], (it / C::kStages) & 1, ctx, kWaitBwdDkDv + 2)) { ok = false; break; }
                    const uint32_t aQ = smem_u32(sStage + st * C::kStageBytes);
                    const uint32_t dQ = desc_lo_k_major(aQ), dDO = desc_lo_k_major(aQ + C::kSubTileBytes);
                    const uint32_t tS = tmem_base + kColS;
                    if (!kVInTmem && x == 0 && !mbar_wait_uniform(&bars->v_full, k & 1, ctx, kWaitBwdDkDv + 3)) { ok = false; break; }
                    if (it >= 1 && !mbar_wait_uniform(&bars->s_free, (it - 1) & 1, ctx, kWaitBwdDkDv + 9)) { ok = false; break; }
                    if (kPBufs > 1 && it >= kPBufs && !mbar_wait_uniform(&bars->p_free[it % kPBufs], ((it / kPBufs) & 1) ^ 1, ctx, kWaitBwdDkDv + 8)) { ok = false; break; }
                    tc_fence_after();
                    if (elect_one()) {
                        mbar_arrive(&bars->s_full);  // (the phase of the step before was over when s_free was)
#pragma unroll
                        for (int kk = 0; kk < HD / 16; ++kk)
                            if constexpr (kVInTmem) mma_ts(tP, tVt + 8 * kk, dDO + desc_step_k_major(kk, C::kSubBoxBytes), idesc_sc, kk > 0);
                            else mma_ss(tP, dV + desc_step_k_major(kk, C::kBigBoxBytes), dDO + desc_step_k_major(kk, C::kSubBoxBytes), idesc_sc, kk > 0);
                        if (!kVInTmem && last) mma_commit(&bars->v_empty);
#pragma unroll
                        for (int kk = 0; kk < HD / 16; ++kk)
                            mma_ts(tS, tKt + 8 * kk, dQ + desc_step_k_major(kk, C::kSubBoxBytes), idesc_sc, kk > 0);
                        mma_commit(&bars->s_full);
                        if (last) mma_commit(&bars->s_done);
                    }
                    __syncwarp();
                }
            }
            if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&bars->abort_flag) != 0)) {
                if (elect_one()) {
                    mma_commit(&bars->drain2);
                    mbar_wait_drain(&bars->drain2, 0);
                }
            }
            __syncwarp();
        } else if (warp == 2) {
            // ---- gradient MMAs: dV += P^T dO and dK += dS^T Q of step `it`
            constexpr uint32_t idesc_acc = idesc_bf16(128, HD, 0, 1);
            int it = 0;
            bool ok = true;
            for (int k = 0; ok; ++k) {
                DkDvItem t;
                if (!next_item(k, kWaitBwdDkDv + 12, &t)) break;
                const int steps = t.total_steps;
                // the first products of an item overwrite the accumulators: the previous item's must have been read out
                if (k > 0 && !mbar_wait_uniform(&bars->acc_empty, (k - 1) & 1, ctx, kWaitBwdDkDv + 13)) break;
                for (int x = 0; x < steps; ++x, ++it) {
                    const int st = it % C::kStages;
                    const int bf = it % kPBufs;
                    if (!mbar_wait_uniform(&bars->p_full[bf], (it / kPBufs) & 1, ctx, kWaitBwdDkDv + 4)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t aQ = smem_u32(sStage + st * C::kStageBytes);
                    const uint32_t dQmn = desc_lo_mn_major(aQ, C::kSubBoxBytes);
                    const uint32_t dDOmn = desc_lo_mn_major(aQ + C::kSubTileBytes, C::kSubBoxBytes);
                    // the 16 queries of K slice kk: P^T in packed columns [16 kk, +8) of the buffer, dS^T in [16 kk + 8, +8)
                    const uint32_t tPt = tmem_base + kColPdS + bf * 64;
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < kSubTile / 16; ++kk)
                            mma_ts(tmem_base + kColDV, tPt + 16 * kk, dDOmn + kk * kDescStepMn, idesc_acc, (x > 0) || (kk > 0));
#pragma unroll
                        for (int kk = 0; kk < kSubTile / 16; ++kk)
                            mma_ts(tmem_base + kColDK, tPt + 16 * kk + 8, dQmn + kk * kDescStepMn, idesc_acc, (x > 0) || (kk > 0));
                        mma_commit(&bars->st_empty[st]);
                        mma_commit(&bars->p_free[bf]);
                        if (x == steps - 1) mma_commit(&bars->acc_full);
                    }
                    __syncwarp();
                }
            }
            if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&bars->abort_flag) != 0)) {
                if (elect_one()) {
                    mma_commit(&bars->drain);
                    mbar_wait_drain(&bars->drain, 0);
                }
            }
            __syncwarp();
        } else {
            // ---- K and V of every item (and the tensor-memory allocation)
            if (lane == 0) {
                int n_k = 0, n_v = 0;  // K and V tiles requested so far
                for (int k = 0;; ++k) {
                    if (!mbar_wait(&bars->sched_full[k % kSched], (k / kSched) & 1, ctx, kWaitBwdDkDv + 15)) break;
                    const DkDvItem t = bars->item[k % kSched];
                    if (t.total_steps == 0) break;
                    if (k > 0 && !mbar_wait(&bars->kt_full, (k - 1) & 1, ctx, kWaitBwdDkDv + 19)) break;
                    mbar_expect_tx(&bars->k_full, C::kBigTileBytes);
                    for (int bx = 0; bx < C::kBoxes; ++bx)
                        tma_load_4d(sK + bx * C::kBigBoxBytes, &p.tm_k, &bars->k_full, bx * 64, t.hk, t.tk0, t.b);
                    ++n_k;
                    // (where V is copied as well, the wait for kt_full stands for both)
                    if (!kVInTmem && k > 0 && !mbar_wait(&bars->v_empty, (k - 1) & 1, ctx, kWaitBwdDkDv + 20)) break;
                    mbar_expect_tx(&bars->v_full, C::kBigTileBytes);
                    for (int bx = 0; bx < C::kBoxes; ++bx)
                        tma_load_4d(sV + bx * C::kBigBoxBytes, &p.tm_v, &bars->v_full, bx * 64, t.hk, t.tk0, t.b);
                    ++n_v;
                }
                if (bars->abort_flag != 0) {
                    if (n_k > 0) mbar_wait_drain(&bars->k_full, (n_k - 1) & 1);
                    if (n_v > 0) mbar_wait_drain(&bars->v_full, (n_v - 1) & 1);
                }
            }
            __syncwarp();
        }
    } else if (warp < 12) {
        // ---- elementwise.  Thread (quad, lane, group) owns key row 32 quad + lane and the query columns
        // [32 group, +32) of every step.  (Letting the two groups of four warps take alternate steps with a
        // whole row per thread was measured in an earlier form with two S^T buffers: the chain S^T ->
        // elementwise -> gradient MMAs is what a step waits for, and half the columns per thread halve its
        // elementwise part: 3.33 against 3.53 ms on the Llama2-7B 32k shape.)
        setmaxnreg_inc<C::kRegsElem>();
        const int quad = warp & 3;
        const int group = (warp - 4) >> 2;
        const int row = quad * 32 + lane;  // key row of the tile owned by this thread
        const uint32_t t_row = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
        const float c2 = p.scale_log2;
        bool ok = true;
        int it = 0;
        auto lds4 = [](uint32_t a) {
            // explicit shared-memory loads: through a generic pointer they cost far more latency
            float4 r;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "r"(a));
            return r;
        };
        for (int k = 0; ok; ++k) {
            DkDvItem t;
            if (!next_item(k, kWaitBwdDkDv + 14, &t)) break;
            const bool key_valid = row < t.k_valid;  // rows past the end of a ragged tile belong to other tiles
            const int hq0 = t.hk * rep;
            for (int hq = hq0; ok && hq < hq0 + rep; ++hq) {
                const HeadWalk w = head_walk(geo, hq, t.tk0);
                // where this thread's dS^T values go when they are spilled: key row `row` of block (j, n) of the
                // spill unit (b, hq, g).  A block is stored chunk-major (16-byte chunk c of row r at uint4 index
                // c * 128 + r), so the 32 lanes of a warp write 512 contiguous bytes at a time.
                uint4* spill_head = nullptr;
                if constexpr (kSpill) {
                    const long long su = (static_cast<long long>(t.b) * (p.pass.nk * rep) + (hq - p.pass.hk0 * rep)) * geo.groups + w.g;
                    spill_head = reinterpret_cast<uint4*>(p.spill + spill_block(su, Tg, w.j, w.n_begin) * kSpillBlockElems) + row;
                }
                for (int n = w.n_begin; n < w.n_end; ++n, ++it) {
                    const int cg0 = 2 * group;   // first 16-column chunk of this thread
                    const int st = it % C::kStages;
                    // The statistics of this step travel with its stage; the score MMA warp's arrival on s_full says that
                    // it has seen the stage land.  (Every wait here is 5 % of a step with head size 64.)
                    if (!mbar_wait_uniform(&bars->s_full, it & 1, ctx, kWaitBwdDkDv + 6)) { ok = false; break; }
                    tc_fence_after();
                    // copy this thread's part of dP^T and S^T into registers and release their buffers as soon as the
                    // copies have landed, so that the score products of the next step run while this one is worked on
                    uint32_t pr[kCols];
                    tmem_ld_32x32(t_row + kColP + 16 * cg0, pr);
                    uint32_t sbuf[2][16];
                    tmem_ld_32x16(t_row + kColS + 16 * cg0, sbuf[0]);
                    tmem_ld_32x16(t_row + kColS + 16 * (cg0 + 1), sbuf[1]);
                    tmem_wait_ld();
                    tc_fence_before();
                    mbar_arrive_warp(&bars->s_free);
                    const uint32_t stat_sa = smem_u32(sStat + st * 2 * kSubTile);  // lse[64] then D[64] of this stage
                    // query x of this sub-tile sees key row r iff x is a valid row of the sub-tile and, in the
                    // diagonal tile, 128 j + r <= 64 n + x
                    const int q_valid = subtile_ref(w.L, n).valid;
                    const bool diagonal = n < w.n_begin + 2;
                    const bool masked = diagonal || q_valid < kSubTile;
                    uint4* spill_dst = nullptr;
                    if constexpr (kSpill) spill_dst = spill_head + static_cast<size_t>(n - w.n_begin) * (kSpillBlockElems / 8);
                    uint32_t pk[kChunks][2][8];  // bf16 P^T and dS^T
                    // P^T of chunk cg goes to the packed columns [16 cg, +8), dS^T to [16 cg + 8, +8): at once where
                    // there are two buffers (the score MMAs of this step were held back until this one was free),
                    // else at the end of the step, when the gradient MMAs of the step before are done with it
                    const int bf = it % kPBufs;
                    const uint32_t tPdS = t_row + kColPdS + bf * 64 + 16 * cg0;
                    auto store_chunk = [&](int c) {
                        tmem_st_32x8(tPdS + 16 * c, pk[c][0]);
                        tmem_st_32x8(tPdS + 16 * c + 8, pk[c][1]);
                    };
                    // 16 queries of this thread's key row, two columns per instruction for the multiply-adds
                    auto weights = [&](int c) {
                        const uint64_t c2x2 = f2_pack(c2, c2), nl2e = f2_pack(-kLog2e, -kLog2e);
#pragma unroll
                        for (int e4 = 0; e4 < 4; ++e4) {
                            const float4 l = lds4(stat_sa + (16 * (cg0 + c) + 4 * e4) * 4);
                            const float4 dd = lds4(stat_sa + kSubTile * 4 + (16 * (cg0 + c) + 4 * e4) * 4);
                            const uint64_t lp[2] = {f2_pack(l.x, l.y), f2_pack(l.z, l.w)};
                            const uint64_t dp[2] = {f2_pack(dd.x, dd.y), f2_pack(dd.z, dd.w)};
#pragma unroll
                            for (int u = 0; u < 2; ++u) {
                                const int e = 4 * e4 + 2 * u;   // column within the chunk
                                const int x = 16 * c + e;       // column among this thread's
                                const uint64_t xs = f2_fma(f2_pack(__uint_as_float(sbuf[c][e]), __uint_as_float(sbuf[c][e + 1])), c2x2,
                                                           f2_mul(lp[u], nl2e));
                                float x0, x1;
                                f2_unpack(xs, x0, x1);
                                const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
                                pk[c][0][e >> 1] = pack_bf16(p0, p1);
                                const uint64_t tt = f2_sub(f2_pack(__uint_as_float(pr[x]), __uint_as_float(pr[x + 1])), dp[u]);
                                float d0, d1;
                                f2_unpack(f2_mul(f2_pack(p0, p1), tt), d0, d1);
                                pk[c][1][e >> 1] = pack_bf16(d0, d1);
                            }
                        }
                    };
                    auto hand_on = [&](int c) {
                        if constexpr (kPBufs > 1) store_chunk(c);
                        if constexpr (kSpill) {
                            // streaming stores: written once, read once by the dQ kernel much later
#pragma unroll
                            for (int cc = 0; cc < 2; ++cc) {
                                uint4 x = make_uint4(pk[c][1][4 * cc], pk[c][1][4 * cc + 1], pk[c][1][4 * cc + 2], pk[c][1][4 * cc + 3]);
                                if (!key_valid) x = make_uint4(0u, 0u, 0u, 0u);
                                __stcs(spill_dst + (2 * (cg0 + c) + cc) * kTile, x);
                            }
                        }
                    };
                    // Of the 32 x 32 entries of a warp on the diagonal tile, all are visible, none, or those on one side of
                    // their own diagonal.
                    auto masked_weights = [&](int c) {
                        const int none = diagonal ? quad * 32 - (n & 1) * kSubTile : -kSubTile;  // queries before it see no key row of the warp
                        const int x0 = 16 * (cg0 + c);
                        if (x0 + 15 < none || x0 >= q_valid) {
#pragma unroll
                            for (int e = 0; e < 8; ++e) pk[c][0][e] = pk[c][1][e] = 0u;
                            return;
                        }
                        weights(c);
                        if (x0 >= none + 31 && x0 + 16 <= q_valid) return;
                        // A masked entry is cleared in the packed result, never multiplied by zero: statistics of rows
                        // that are not valid were never loaded.
                        const int first = (diagonal ? none + lane : 0) - x0, end = q_valid - x0;  // visible columns
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const uint32_t keep = (2 * e >= first && 2 * e < end ? 0x0000ffffu : 0u) | (2 * e + 1 >= first && 2 * e + 1 < end ? 0xffff0000u : 0u);
                            pk[c][0][e] &= keep, pk[c][1][e] &= keep;
                        }
                    };
                    // One branch for the step, so that both chunks of an unmasked step are one run of instructions: with a branch in
                    // each chunk, and every entry of a masked step compared and selected, a launch took 33.1 instead of 30.3 us
                    // on 4 x 2000 tokens in groups of 200 (head size 64), 101 instead of 98 on 2 x 4096 tokens grouped query,
                    // 2490 instead of 2405 at head size 64 and 32k, 380,000 instead of 375,000 clocks on Llama2-7B 8k (at the
                    // power limit, the same time).
                    if (masked) {
#pragma unroll
                        for (int c = 0; c < kChunks; ++c) masked_weights(c), hand_on(c);
                    } else {
#pragma unroll
                        for (int c = 0; c < kChunks; ++c) weights(c), hand_on(c);
                    }
                    if constexpr (kPBufs == 1) {
                        if (it >= 1 && !mbar_wait_uniform(&bars->p_free[0], (it - 1) & 1, ctx, kWaitBwdDkDv + 8)) { ok = false; break; }
                        tc_fence_after();
#pragma unroll
                        for (int c = 0; c < kChunks; ++c) store_chunk(c);
                    }
                    tmem_wait_st();
                    tc_fence_before();
                    mbar_arrive_warp(&bars->p_full[bf]);
                }
            }
        }
    } else {
        // ---- epilogue: the copies of K and V into tensor memory and the read-out of the accumulators
        setmaxnreg_dec<C::kRegsOther>();
        const int quad = warp & 3;
        const int row = quad * 32 + lane;
        const uint32_t t_row = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
        uint8_t* stage = sOut + quad * 8192;
        uint32_t used = 0;
        // K of item k goes from its shared-memory tile into tensor memory, where it is the A operand of
        // S^T = K Q^T, and where HD = 64 leaves room V, the A operand of dP^T = V dO^T: an A operand in shared memory would be read again by every step (4 KB per MMA
        // against 2 KB of B), and shared-memory bandwidth is what bounds this kernel.  One key row per thread:
        // the 16-byte chunks of the 128-byte-swizzled rows, 32 packed columns for each 64 values.
        auto copy_operands = [&](int k) -> bool {
            if (!mbar_wait_uniform(&bars->k_full, k & 1, ctx, kWaitBwdDkDv + 17)) return false;
            if (k > 0 && !mbar_wait_uniform(&bars->s_done, (k - 1) & 1, ctx, kWaitBwdDkDv + 21)) return false;
            tc_fence_after();
            auto copy_row = [&](const uint8_t* tile, uint32_t t_addr) {
#pragma unroll
                for (int bx = 0; bx < C::kBoxes; ++bx) {
                    const uint32_t src = smem_u32(tile) + bx * C::kBigBoxBytes + row * 128;
                    uint32_t kr[32];
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                                     : "=r"(kr[4 * c]), "=r"(kr[4 * c + 1]), "=r"(kr[4 * c + 2]), "=r"(kr[4 * c + 3])
                                     : "r"(src + ((c ^ (row & 7)) << 4)));
                    }
                    tmem_st_32x32(t_addr + bx * 32, kr);
                }
            };
            copy_row(sK, t_row + kColKt);
            if constexpr (kVInTmem) {
                // (a warp that gives up must leave no store to tensor memory behind; waiting for V ahead of K's copy as well
                // takes half a percent longer on groups of 384)
                if (!mbar_wait_uniform(&bars->v_full, k & 1, ctx, kWaitBwdDkDv + 3)) { tmem_wait_st(); return false; }
                copy_row(sV, t_row + kColVt);
            }
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive_warp(&bars->kt_full);
            return true;
        };
        DkDvItem next;
        bool more = next_item(0, kWaitBwdDkDv + 18, &next) && copy_operands(0);
        for (int k = 0; more; ++k) {
            const DkDvItem t = next;
            // the operands of the next item, if there is one, as soon as this item's score products are done
            more = next_item(k + 1, kWaitBwdDkDv + 18, &next);
            if (more && !copy_operands(k + 1)) break;
            if (!mbar_wait_uniform(&bars->acc_full, k & 1, ctx, kWaitBwdDkDv + 7)) break;
            tc_fence_after();
            const size_t out_row = (static_cast<size_t>(t.b) * geo.N + t.tk0 + row) * p.dkv_tok_stride + static_cast<size_t>(t.hk) * HD;
            const int tok0 = t.tk0 + quad * 32, valid = t.k_valid - quad * 32;
            store_acc_rows<HD>(&p.tm_dv, stage, used, t_row + kColDV, 1.0f, p.dv + out_row, t.hk, tok0, t.b, valid, [] {});
            store_acc_rows<HD>(&p.tm_dk, stage, used, t_row + kColDK, p.scale, p.dk + out_row, t.hk, tok0, t.b, valid, [&] {
                tc_fence_before();
                mbar_arrive_warp(&bars->acc_empty);
            });
        }
        if (lane == 0) bulk_wait_all();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 3) {
        tc_fence_after();
        tmem_dealloc(tmem_base, C::kTmemCols);
    }
}

// ------------------------------------------------------------------------------------------------
// 4. dQ from spilled dS^T
// ------------------------------------------------------------------------------------------------
// dQ_i = scale * sum_j dS_ij K_j over the key tiles j_begin..i of the group, with dS_ij read back from
// the blocks the spilling dK,dV kernel wrote: nothing is recomputed, the kernel is a chain of
// 128x128x128 products whose A operand streams from global memory once (memory bound).
//
// Persistent: one CTA per SM takes pairs of neighbouring query tiles of a unit, heaviest first, by cluster
// launch control.  The two tiles of a pair share the K tiles they stream: 48 instead of 64 KB through L2
// and shared memory for every product.  Warp 0 draws the items and loads with TMA (it runs ahead across item boundaries,
// so the ring never drains between items), warp 1 issues the MMAs into one of two pairs of accumulators in
// tensor memory, warps 2-5 write the finished accumulators out while the next item is being multiplied.
// Bound by reading dS (8.7 GB on Llama2-7B 32k: 1.33 ms at the measured copy rate, 1.50 taken; a tile at a time
// took 1.60).
// A block (j, n) is copied to shared memory as it lies in global memory (one bulk copy for the blocks
// (j, 2i) and (j, 2i+1), which are neighbours): chunk-major, i.e. the 16-byte chunk c (8 queries) of
// key row r at byte (c * 128 + r) * 16.  Eight key rows of one chunk are 128 contiguous bytes: the
// "core matrix" of an MN-major operand without swizzle (M = queries, K = keys), with 2048 bytes
// between chunks along M and 128 bytes between groups of 8 keys along K; the two blocks side by side
// are the 128-query A operand.  B is the K tile, MN-major (N = d) with the 128-byte swizzle TMA
// leaves, as in the recomputing dQ kernel.
template <int HD>
struct DqSpillCfg {
    static constexpr int kThreads = 192;  // TMA warp, MMA warp, four epilogue warps
    static constexpr int kBoxes = HD / 64;
    static constexpr int kKBoxBytes = kTile * 128;
    static constexpr int kKBytes = kBoxes * kKBoxBytes;
    static constexpr int kDsBytes = 2 * kSpillBlockElems * 2;  // dS of one query tile against one key tile
    static constexpr int kSlotBytes = 32768;                   // a K tile or a dS tile
    static_assert(kKBytes <= kSlotBytes && kDsBytes <= kSlotBytes, "slot size");
    static constexpr int kRing = 6;   // K_j, dS_1j, dS_0j, K_{j+1}, ...
    static constexpr int kSched = 8;  // work items the producer can be ahead of the epilogue: at most 5
    static constexpr int kOutBytes = 4 * 2 * 4096;
    static constexpr int kBarBytes = 1024;
    static constexpr int kSmemBytes = kRing * kSlotBytes + kOutBytes + kBarBytes;
    static constexpr int kTmemCols = 512;  // two pairs of accumulators of 128 columns
};

struct DqSpillItem {
    int b, h, hk;
    long long unit;
    GroupLayout L;
    TilePair t;
};
struct DqSpillBars {
    uint64_t full[6], empty[6];
    uint64_t acc_full[2], acc_empty[2];
    uint64_t sched_full[8];
    uint64_t drain, clc;
    alignas(16) uint8_t clc_resp[16];
    DqSpillItem item[8];  // b = -1: no more items
    uint32_t tmem_slot;
    int abort_flag;
};
static_assert(sizeof(DqSpillBars) <= 1024, "barrier block");

// Work item `id`: a pair of query tiles, the heaviest of a chunk of units first, as in the other kernels.
// Units are taken from the last one down: the dS^T that was written last may still be in L2.  false marks
// a slot of a group that has fewer pairs than the largest one.
__device__ __forceinline__ bool dq_spill_item(const BwdDqSpillParams& p, int id, DqSpillItem* w) {
    const Geometry& geo = p.geo;
    int unit, rank, g;
    p.order.decode(id, &unit, &rank);
    unit = p.order.units - 1 - unit;
    w->b = p.by_heads(geo.by_groups(unit, &g), &w->h);
    w->h += p.pass.hk0 * geo.rep;
    w->hk = geo.by_rep(w->h);
    w->unit = unit;
    w->L = group_layout(geo, (w->h < geo.n_unshifted) ? 0 : geo.shift, g);
    if (rank >= pairs_of_group(w->L, p.single)) return false;
    w->t = tile_pair(w->L, rank, p.single);
    return true;
}

template <int HD>
__global__ void __launch_bounds__(DqSpillCfg<HD>::kThreads, 1) s2a_bwd_dq_spill_kernel(const __grid_constant__ BwdDqSpillParams p) {
    using C = DqSpillCfg<HD>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = smem_raw;  // 1024-byte aligned: nothing precedes the dynamic array
    uint8_t* sOut = smem + C::kRing * C::kSlotBytes;
    DqSpillBars* bars = reinterpret_cast<DqSpillBars*>(sOut + C::kOutBytes);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    const int Tg = p.geo.tiles_per_group;

    if (threadIdx.x == 0) {
        for (int x = 0; x < C::kRing; ++x) {
            mbar_init(&bars->full[x], 1);
            mbar_init(&bars->empty[x], 1);
        }
        for (int x = 0; x < 2; ++x) {
            mbar_init(&bars->acc_full[x], 1);
            mbar_init(&bars->acc_empty[x], 4);  // one arrival per epilogue warp
        }
        for (int x = 0; x < C::kSched; ++x) mbar_init(&bars->sched_full[x], 1);
        mbar_init(&bars->drain, 1);
        mbar_init(&bars->clc, 1);
        fence_barrier_init();
        tma_prefetch_desc(&p.tm_k);
        tma_prefetch_desc(&p.tm_dq);
    }
    if (warp == 1) {
        tmem_alloc(&bars->tmem_slot, C::kTmemCols);
        tmem_relinquish();
    }
    wait_for_predecessor();
    // A bounded wait that expired earlier (in any kernel) leaves the status word set: later CTAs
    // then return at once instead of each running into its own time limit.
    if (threadIdx.x == 0) bars->abort_flag = *reinterpret_cast<volatile int*>(p.status);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    release_successor();
    const uint32_t tmem_base = bars->tmem_slot;
    if (bars->abort_flag != 0) {
        if (warp == 1) tmem_dealloc(tmem_base, C::kTmemCols);
        return;
    }
    const WaitCtx ctx{&bars->abort_flag, p.status, p.host_status};
    auto next_item = [&](int k, int where, DqSpillItem* w) -> bool {
        if (!mbar_wait_uniform(&bars->sched_full[k % C::kSched], (k / C::kSched) & 1, ctx, where)) return false;
        *w = bars->item[k % C::kSched];
        return w->b >= 0;
    };

    if (warp == 0) {
        // ---- work items + TMA producer ------------------------------------------------------------
        if (lane == 0) {
            uint32_t x = 0;  // ring slots filled so far
            bool ok = true;
            ItemSource items{&bars->clc, bars->clc_resp};
            int id = static_cast<int>(blockIdx.x);
            auto slot = [&](uint32_t bytes) -> uint8_t* {
                const uint32_t st = x % C::kRing;
                if (!mbar_wait(&bars->empty[st], ((x / C::kRing) & 1) ^ 1, ctx, kWaitBwdDqSpill + 1)) {
                    ok = false;
                    return nullptr;
                }
                mbar_expect_tx(&bars->full[st], bytes);
                return smem + st * C::kSlotBytes;
            };
            for (int k = 0; ok; ++k) {
                DqSpillItem w;
                while (id >= 0 && !dq_spill_item(p, id, &w)) {  // skip the empty slots of smaller groups
                    id = items.next(ctx, kWaitBwdDqSpill + 7, &ok);
                }
                if (id < 0) w.b = -1;
                bars->item[k % C::kSched] = w;
                mbar_arrive(&bars->sched_full[k % C::kSched]);  // release: the item is visible to whoever sees the phase
                if (id < 0) break;
                for (int n = 0; ok && n < w.t.n[1]; ++n) {
                    const int j = w.t.j_begin + n;
                    const int tk0 = tile_ref(w.L, j).tok0;
                    uint8_t* dst = slot(C::kKBytes);
                    if (!ok) break;
                    for (int bx = 0; bx < C::kBoxes; ++bx)
                        tma_load_4d(dst + bx * C::kKBoxBytes, &p.tm_k, &bars->full[x % C::kRing], bx * 64, w.hk, tk0, w.b);
                    ++x;
                    for (int t = 1; t >= 0 && n < w.t.n[t]; --t) {
                        dst = slot(C::kDsBytes);
                        if (!ok) break;
                        bulk_load_1d(dst, p.spill + spill_block(w.unit, Tg, j, 2 * w.t.i[t]) * kSpillBlockElems, C::kDsBytes,
                                     &bars->full[x % C::kRing]);
                        ++x;
                    }
                }
                if (ok) id = items.next(ctx, kWaitBwdDqSpill + 7, &ok);
            }
            if (bars->abort_flag != 0) {
                for (uint32_t y = (x > C::kRing ? x - C::kRing : 0); y < x; ++y)
                    mbar_wait_drain(&bars->full[y % C::kRing], (y / C::kRing) & 1);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---- MMA issuer (warp-uniform loop, one elected lane issues) ------------------------------
        constexpr uint32_t idesc = idesc_bf16(128, HD, 1, 1);
        uint32_t x = 0;
        bool ok = true;
        auto wait_slot = [&](uint32_t y) -> bool {
            return mbar_wait_uniform(&bars->full[y % C::kRing], (y / C::kRing) & 1, ctx, kWaitBwdDqSpill + 4);
        };
        for (int k = 0; ok; ++k) {
            DqSpillItem w;
            if (!next_item(k, kWaitBwdDqSpill + 2, &w)) break;
            const int buf = k & 1;
            if (!mbar_wait_uniform(&bars->acc_empty[buf], ((k >> 1) & 1) ^ 1, ctx, kWaitBwdDqSpill + 3)) break;
            for (int n = 0; ok && n < w.t.n[1]; ++n) {
                const uint32_t xk = x++;
                ok = wait_slot(xk);
                const uint32_t dB = desc_lo_mn_major(smem_u32(smem + (xk % C::kRing) * C::kSlotBytes), C::kKBoxBytes);
#pragma unroll 1
                for (int t = 1; ok && t >= 0; --t) {
                    const int n_t = t ? w.t.n[1] : w.t.n[0];
                    if (n >= n_t) break;
                    const uint32_t xd = x++;
                    ok = wait_slot(xd);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t dA = desc_lo_mn_major_plain(smem_u32(smem + (xd % C::kRing) * C::kSlotBytes), 128);
                    const uint32_t tAcc = tmem_base + buf * 256 + t * 128;
                    const bool last_t = t == 0 || n >= w.t.n[0];  // last product with this K tile
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < kTile / 16; ++kk)
                            mma_ss_hi(tAcc, dA + kk * (256u >> 4), desc_hi_plain(2048), dB + kk * kDescStepMn, kDescHi, idesc,
                                      (n > 0) || (kk > 0));
                        mma_commit(&bars->empty[xd % C::kRing]);
                        if (last_t) mma_commit(&bars->empty[xk % C::kRing]);
                        if (last_t && n == w.t.n[1] - 1) mma_commit(&bars->acc_full[buf]);
                    }
                    __syncwarp();
                }
            }
        }
        if (__any_sync(0xffffffffu, *reinterpret_cast<volatile int*>(&bars->abort_flag) != 0)) {
            if (elect_one()) {
                mma_commit(&bars->drain);
                mbar_wait_drain(&bars->drain, 0);
            }
        }
        __syncwarp();
    } else {
        // ---- epilogue: thread owns accumulator row 32 * quad + lane -------------------------------
        const int quad = warp & 3;
        const int row = quad * 32 + lane;
        const uint32_t t_row = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
        uint8_t* stage = sOut + quad * 8192;
        uint32_t used = 0;
        for (int k = 0;; ++k) {
            DqSpillItem w;
            if (!next_item(k, kWaitBwdDqSpill + 5, &w)) break;
            const int buf = k & 1;
            if (!mbar_wait_uniform(&bars->acc_full[buf], (k >> 1) & 1, ctx, kWaitBwdDqSpill + 6)) break;
            tc_fence_after();
#pragma unroll 1
            for (int t = w.t.n[0] > 0 ? 0 : 1; t < 2; ++t) {
                const TileRef tq = tile_ref(w.L, t ? w.t.i[1] : w.t.i[0]);
                __nv_bfloat16* dst = p.dq + (static_cast<size_t>(w.b) * p.geo.N + tq.tok0 + row) * p.dq_tok_stride + static_cast<size_t>(w.h) * HD;
                store_acc_rows<HD>(&p.tm_dq, stage, used, t_row + buf * 256 + t * 128, p.scale, dst, w.h, tq.tok0 + quad * 32, w.b,
                                   tq.valid - quad * 32, [&] {
                                       if (t == 1) {
                                           tc_fence_before();
                                           mbar_arrive_warp(&bars->acc_empty[buf]);
                                       }
                                   });
            }
        }
        if (lane == 0) bulk_wait_all();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, C::kTmemCols);
    }
}

}  // namespace

namespace {
// The kernels place their tiles from the start of the dynamic array, and the register split of the dK,dV
// kernel draws on what a block is launched with (min_regs).
template <typename Kernel>
cudaError_t configure_one(Kernel kernel, int smem_bytes, int min_regs) {
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, kernel);
    if (e != cudaSuccess) return e;
    if (a.numRegs < min_regs || a.sharedSizeBytes != 0) return cudaErrorInvalidConfiguration;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
}
template <int HD>
cudaError_t configure_all() {
    cudaError_t e = configure_one(s2a_bwd_dq_kernel<HD>, DqCfg<HD>::kSmemBytes, DqCfg<HD>::kRegsLaunch);
    if (e == cudaSuccess) e = configure_one(s2a_bwd_dkdv_kernel<HD, false>, BwdCfg<HD>::kSmemBytes, BwdCfg<HD>::kRegsLaunch);
    if (e == cudaSuccess) e = configure_one(s2a_bwd_dkdv_kernel<HD, true>, BwdCfg<HD>::kSmemBytes, BwdCfg<HD>::kRegsLaunch);
    if (e == cudaSuccess) e = configure_one(s2a_bwd_dq_spill_kernel<HD>, DqSpillCfg<HD>::kSmemBytes, 0);
    return e;
}
}  // namespace

cudaError_t configure_bwd() {
    const cudaError_t e = configure_all<64>();
    return e != cudaSuccess ? e : configure_all<128>();
}

cudaError_t launch_bwd_preprocess(const PreParams& p, int d, cudaStream_t stream, bool overlap) {
    const int rows_per_block = 256 / (d / 8) * kPreRows;
    const unsigned grid = static_cast<unsigned>((p.rows + rows_per_block - 1) / rows_per_block);
    return d == 64 ? launch_kernel(s2a_bwd_preprocess_kernel<64>, grid, 256, 0, stream, p, overlap)
                   : launch_kernel(s2a_bwd_preprocess_kernel<128>, grid, 256, 0, stream, p, overlap);
}

cudaError_t launch_bwd_dq(const BwdDqParams& p, int d, cudaStream_t stream, bool overlap) {
    const Geometry& g = p.geo;
    const unsigned grid = static_cast<unsigned>(static_cast<long long>(g.B) * g.H * g.groups * g.tiles_per_group);
    return d == 64 ? launch_kernel(s2a_bwd_dq_kernel<64>, grid, DqCfg<64>::kThreads, DqCfg<64>::kSmemBytes, stream, p, overlap)
                   : launch_kernel(s2a_bwd_dq_kernel<128>, grid, DqCfg<128>::kThreads, DqCfg<128>::kSmemBytes, stream, p, overlap);
}

namespace {
template <int HD>
cudaError_t launch_dkdv(const BwdDkDvParams& p, unsigned grid, cudaStream_t stream) {
    return p.spill != nullptr ? launch_kernel(s2a_bwd_dkdv_kernel<HD, true>, grid, BwdCfg<HD>::kThreads, BwdCfg<HD>::kSmemBytes, stream, p, false)
                              : launch_kernel(s2a_bwd_dkdv_kernel<HD, false>, grid, BwdCfg<HD>::kThreads, BwdCfg<HD>::kSmemBytes, stream, p, false);
}
}  // namespace

cudaError_t launch_bwd_dkdv(const BwdDkDvParams& p, int d, cudaStream_t stream) {
    const Geometry& g = p.geo;
    const unsigned grid = static_cast<unsigned>(static_cast<long long>(g.B) * p.pass.nk * g.groups * g.tiles_per_group);
    return d == 64 ? launch_dkdv<64>(p, grid, stream) : launch_dkdv<128>(p, grid, stream);
}

cudaError_t launch_bwd_dq_spill(const BwdDqSpillParams& p, int d, cudaStream_t stream, bool overlap) {
    const Geometry& g = p.geo;
    const unsigned grid = static_cast<unsigned>(static_cast<long long>(g.B) * p.pass.nk * (g.H / g.Hkv) * g.groups * p.pairs_per_group);
    return d == 64 ? launch_kernel(s2a_bwd_dq_spill_kernel<64>, grid, DqSpillCfg<64>::kThreads, DqSpillCfg<64>::kSmemBytes, stream, p, overlap)
                   : launch_kernel(s2a_bwd_dq_spill_kernel<128>, grid, DqSpillCfg<128>::kThreads, DqSpillCfg<128>::kSmemBytes, stream, p, overlap);
}

}  // namespace s2a
