// Host side of the C-ABI declared in include/s2a.h: argument validation, TMA tensor maps,
// kernel launches.  Nothing here allocates device memory.
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <mutex>

#include "../../include/s2a.h"
#include "host_plan.h"
#include "s2a_params.h"
#include "sm100_ptx.cuh"

namespace s2a {
namespace {

// Device-wide status word written by kernels whose bounded wait expired (one copy per device
// that loads this library).
__device__ int g_status_word;

// Host-visible mirrors of the status words, one per device (64 bytes apart): page-locked and mapped
// into the device address space, so that a kernel can store the code of an expired wait where the
// next entry point sees it without synchronising.  This is ordinary static memory, pinned in place
// once per process; nothing is allocated.
constexpr int kMirrorStride = 16;  // ints
constexpr int kMaxDevicesMirror = 64;
alignas(4096) int g_host_status[kMaxDevicesMirror * kMirrorStride];
bool g_host_status_registered = false;

thread_local int tl_last_cuda_error = 0;

constexpr int kMaxDevices = 64;
struct DeviceState {
    bool ready = false;
    int* status_ptr = nullptr;        // device address of g_status_word
    volatile int* host_word = nullptr;  // this device's mirror, host address
    int* host_word_dev = nullptr;     // the same word as the device sees it
    int n_sm = 0;                     // multiprocessors
    // s2a_fwd_bwd_host only: copy streams and the events that order them against the caller's stream
    bool host_path_ready = false;
    cudaStream_t copy_in = nullptr, copy_out = nullptr;
    cudaEvent_t ev_start = nullptr, ev_done = nullptr, ev_in_done = nullptr;
    cudaEvent_t ev_qkv = nullptr, ev_do = nullptr, ev_fwd = nullptr, ev_bwd = nullptr;  // recorded again for every chunk
    std::mutex host_path;  // held by the call that enqueues: its events must not be recorded by another one in between
};
DeviceState g_dev[kMaxDevices];
static_assert(kMaxDevices == kMaxDevicesMirror, "one mirror word per device");
std::mutex g_dev_mutex;  // guards the one-time set-up of a DeviceState (calls may come from several host threads)

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;

int cuda_fail(cudaError_t e) {
    tl_last_cuda_error = static_cast<int>(e);
    return S2A_ERR_CUDA;
}

// Per-device set-up: architecture check, shared-memory attributes, address of the status word.
int prepare_device(DeviceState** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e);
    if (dev < 0 || dev >= kMaxDevices) return S2A_ERR_UNSUPPORTED;
    DeviceState& ds = g_dev[dev];
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    if (!ds.ready) {
        int major = 0;
        e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
        if (e != cudaSuccess) return cuda_fail(e);
        if (major != 10) return S2A_ERR_UNSUPPORTED;
        e = cudaDeviceGetAttribute(&ds.n_sm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return cuda_fail(e);
        if (!g_encode) {
            void* fn = nullptr;
            cudaDriverEntryPointQueryResult qres;
            e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
            if (e != cudaSuccess) return cuda_fail(e);
            if (qres != cudaDriverEntryPointSuccess || !fn) return cuda_fail(cudaErrorNotSupported);
            g_encode = reinterpret_cast<EncodeTiledFn>(fn);
        }
        e = configure_fwd();
        if (e != cudaSuccess) return cuda_fail(e);
        e = configure_bwd();
        if (e != cudaSuccess) return cuda_fail(e);
        e = cudaGetSymbolAddress(reinterpret_cast<void**>(&ds.status_ptr), g_status_word);
        if (e != cudaSuccess) return cuda_fail(e);
        if (!g_host_status_registered) {
            e = cudaHostRegister(g_host_status, sizeof g_host_status, cudaHostRegisterPortable | cudaHostRegisterMapped);
            if (e != cudaSuccess) return cuda_fail(e);
            g_host_status_registered = true;
        }
        ds.host_word = &g_host_status[dev * kMirrorStride];
        e = cudaHostGetDevicePointer(reinterpret_cast<void**>(&ds.host_word_dev), const_cast<int*>(ds.host_word), 0);
        if (e != cudaSuccess) return cuda_fail(e);
        ds.ready = true;
    }
    *out = &ds;
    return S2A_OK;
}

int encode_tmap(CUtensorMap* tm, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides, const cuuint32_t* box) {
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    const CUresult r = g_encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(base), dims, strides, box, estr,
                                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        tl_last_cuda_error = static_cast<int>(cudaErrorInvalidValue);
        return S2A_ERR_CUDA;
    }
    return S2A_OK;
}

// bf16 tensor [B, N, heads, d] viewed as (d, heads, N, B); box = 64 columns x `box_rows` tokens of
// one head, written to shared memory with the 128-byte swizzle the MMA descriptors expect.
// `tok_stride` = elements between consecutive tokens (heads * d when the tensor is dense; 3 * H * d for
// the slices of a packed [B, N, 3, H, d] tensor).
int make_tmap(CUtensorMap* tm, const void* base, int d, int heads, int N, int B, int box_rows, long long tok_stride = 0) {
    if (tok_stride == 0) tok_stride = static_cast<long long>(heads) * d;
    const cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)heads, (cuuint64_t)N, (cuuint64_t)B};
    const cuuint64_t strides[3] = {(cuuint64_t)d * 2, (cuuint64_t)tok_stride * 2, (cuuint64_t)N * tok_stride * 2};
    const cuuint32_t box[4] = {64, 1, (cuuint32_t)box_rows, 1};
    return encode_tmap(tm, base, 4, dims, strides, box);
}

// The same tensor and swizzle with boxes of 64 columns x 128 tokens in the order 0 2 1 3, 4 6 5 7, ... (N % 4 = 0): a
// group of four tokens is two dimensions of two.
int make_tmap_exchanged(CUtensorMap* tm, const void* base, int d, int heads, int N, int B, long long tok_stride = 0) {
    if (tok_stride == 0) tok_stride = static_cast<long long>(heads) * d;
    const cuuint64_t tok = (cuuint64_t)tok_stride * 2;
    const cuuint64_t dims[5] = {(cuuint64_t)heads * d, 2, 2, (cuuint64_t)N / 4, (cuuint64_t)B};
    const cuuint64_t strides[4] = {2 * tok, tok, 4 * tok, N * tok};
    const cuuint32_t box[5] = {64, 2, 2, kTile / 4, 1};
    return encode_tmap(tm, base, 5, dims, strides, box);
}

// variants 2 and 3 of Appendix B exclude each other; no other bits are defined
bool flags_ok(unsigned flags) {
    return (flags & ~static_cast<unsigned>(S2A_FLAG_LEAK_FREE | S2A_FLAG_SWAP_WRAPPED)) == 0 &&
           flags != (S2A_FLAG_LEAK_FREE | S2A_FLAG_SWAP_WRAPPED);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int check_shape(int B, int N, int H, int Hkv, int d, int G, float scale, int n_unshifted, int shift) {
    if (B <= 0 || N <= 0 || H <= 0 || Hkv <= 0 || d <= 0 || G <= 0) return S2A_ERR_INVALID_ARG;
    if (N % G != 0 || H % Hkv != 0) return S2A_ERR_INVALID_ARG;
    if (n_unshifted < 0 || n_unshifted > H) return S2A_ERR_INVALID_ARG;
    if (!(scale > 0.f) || !isfinite(scale)) return S2A_ERR_INVALID_ARG;
    if (shift <= -N || shift >= N) return S2A_ERR_INVALID_ARG;
    if (d != 64 && d != 128) return S2A_ERR_UNSUPPORTED;
    // Every run of tokens of a group must start and end on a multiple of 4 tokens (16 bytes of the
    // fp32 row statistics, which travel by bulk copies); a tensor map wants at least one whole box.
    if (G % 4 != 0 || shift % 4 != 0 || N < kTile) return S2A_ERR_UNSUPPORTED;
    // Ragged tiles (G or shift not a multiple of 128): the key tiles of a KV head follow the partition
    // of its query heads, which must then all have the same shift.
    if ((G % kTile != 0 || shift % kTile != 0) && n_unshifted % (H / Hkv) != 0) return S2A_ERR_UNSUPPORTED;
    // grid sizes and 32-bit token arithmetic
    const long long tiles = (long long)B * H * (N / G) * (G / kTile + 2);
    if (tiles > 0x7fffffffLL || (long long)N + G >= 0x40000000LL) return S2A_ERR_UNSUPPORTED;
    return S2A_OK;
}

// Shape rules of the default entry points (shift G/2 on the second half of the heads).
int check_default_shape(int N, int H, int d, int G) {
    if (d <= 0 || H <= 0 || (H & 1) || (G & 1)) return S2A_ERR_INVALID_ARG;
    if (G % 8 != 0) return (G > 0 && N > 0 && N % G == 0) ? S2A_ERR_UNSUPPORTED : S2A_ERR_INVALID_ARG;
    return S2A_OK;
}

// Largest value of `count` over the groups of both partitions.  All groups of a partition are alike but the
// one that wraps around the end of the sequence, so two of them are looked at however many there are.
template <typename Count>
int most_over_groups(const Geometry& g, Count count) {
    int most = 0;
    const int shifts[2] = {0, g.shift};
    for (int which = 0; which < 2; ++which) {
        if ((which == 0 && g.n_unshifted == 0) || (which == 1 && g.n_unshifted == g.H)) continue;
        const int s = shifts[which], r = ((s % g.G) + g.G) % g.G;
        // the group that starts at token N - G + r: it wraps unless r = 0
        const int wraps = ((g.N - g.G + r - s) / g.G % g.groups + g.groups) % g.groups;
        for (int grp : {wraps, (wraps + 1) % g.groups}) {
            const int n = count(group_layout(g, s, grp));
            if (n > most) most = n;
        }
    }
    return most;
}

Geometry make_geometry(int B, int N, int H, int Hkv, int G, int n_unshifted, int shift, unsigned flags = 0u) {
    Geometry g;
    g.B = B, g.N = N, g.H = H, g.Hkv = Hkv, g.G = G;
    g.n_unshifted = n_unshifted;
    g.shift = shift;
    g.groups = N / G;
    g.leak_free = (flags & S2A_FLAG_LEAK_FREE) ? 1 : 0;
    g.swap_wrapped = (flags & S2A_FLAG_SWAP_WRAPPED) ? 1 : 0;
    g.rep = H / Hkv;
    g.by_group = FastDiv(G), g.by_groups = FastDiv(g.groups), g.by_rep = FastDiv(g.rep);
    // the grid has one slot per (unit, tile rank); groups with fewer tiles leave their last slots idle
    g.tiles_per_group = most_over_groups(g, [](const GroupLayout& L) { return L.nTiles; });
    return g;
}
// Largest number of query tile pairs any group has (see tile_pair).
int most_pairs(const Geometry& g, bool single) {
    return most_over_groups(g, [single](const GroupLayout& L) { return pairs_of_group(L, single); });
}
// Whether the kernels that work on pairs of query tiles take single tiles instead: when the pairs of `heads`
// heads are fewer than the multiprocessors.
bool take_single_tiles(const Geometry& g, int heads, int n_sm) {
    return static_cast<long long>(g.B) * heads * g.groups * most_pairs(g, false) <= n_sm;
}

// Whether launches are so short (some 50 us at most) that starting them early pays, see launch_kernel(): up to
// 32 pairs of a query and a key tile, counted for head size 128, for each multiprocessor.
bool is_short(const Geometry& g, int d, int n_sm) {
    const double T = g.tiles_per_group;
    return static_cast<double>(g.B) * g.H * g.groups * T * (T + 1) / 2 * d / 128 <= 32.0 * n_sm;
}

constexpr float kLog2eHost = 1.4426950408889634f;

// Diagnostic kernel behind s2a_selftest_wait_expiry: one warp waits, with the library's own bounded
// wait and the given limit, on a barrier nothing ever arrives on.  The wait runs out, the expiry is
// reported exactly as a production kernel reports one, and the kernel returns.
constexpr int kWaitSelfTest = 900;
__global__ void __launch_bounds__(32) s2a_wait_selftest_kernel(int* status, int* host_status, long long limit) {
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_flag = 0;
        fence_barrier_init();
    }
    __syncthreads();
    if (*reinterpret_cast<volatile int*>(status) != 0) return;  // like every kernel here: a set status word means "do nothing"
    const WaitCtx ctx{&abort_flag, status, host_status};
    mbar_wait_limit(&bar, 0, ctx, kWaitSelfTest + 1, limit);
}

}  // namespace
}  // namespace s2a

using namespace s2a;

#pragma GCC visibility push(default)
extern "C" {

int s2a_version(void) { return 200; }

int s2a_last_cuda_error(void) { return tl_last_cuda_error; }

const char* s2a_status_string(int status) {
    switch (status) {
        case S2A_OK: return "ok";
        case S2A_ERR_INVALID_ARG: return "invalid argument (null or misaligned pointer, bad size, or workspace too small)";
        case S2A_ERR_UNSUPPORTED: return "unsupported shape or device (need d in {64,128}, G and shift multiples of 4 tokens, N >= 128, sm_100)";
        case S2A_ERR_CUDA: return "a CUDA call failed; see s2a_last_cuda_error()";
        case S2A_ERR_TIMEOUT: return "a bounded device-side wait expired";
        case S2A_ERR_TOO_LARGE: return "B*H*N exceeds the built-in scratch of s2a_bwd_noalloc (see s2a_bwd_noalloc_max_rows)";
        default: return "unknown status";
    }
}

namespace {
// Token strides in elements; 0 means dense ([B, N, heads, d]).
struct TokStrides {
    long long q = 0, kv = 0, dq = 0, dkv = 0;
};

int fwd_impl(const void* q, const void* k, const void* v, void* o, float* lse, int B, int N, int H, int Hkv, int d,
             int G, float scale, int n_unshifted, int shift, unsigned flags, void* stream, const TokStrides& ts) {
    if (!flags_ok(flags)) return S2A_ERR_INVALID_ARG;
    if (!q || !k || !v || !o || !lse) return S2A_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) || !aligned16(lse)) return S2A_ERR_INVALID_ARG;
    int rc = check_shape(B, N, H, Hkv, d, G, scale, n_unshifted, shift);
    if (rc != S2A_OK) return rc;
    DeviceState* ds = nullptr;
    rc = prepare_device(&ds);
    if (rc != S2A_OK) return rc;
    if (*ds->host_word != 0) return S2A_ERR_TIMEOUT;  // an earlier launch gave up: see s2a_device_status()

    FwdParams p;
    memset(&p, 0, sizeof p);
    if ((rc = make_tmap(&p.tm_q, q, d, H, N, B, kTile, ts.q)) != S2A_OK) return rc;
    if ((rc = make_tmap_exchanged(&p.tm_k, k, d, Hkv, N, B, ts.kv)) != S2A_OK) return rc;
    if ((rc = make_tmap(&p.tm_v, v, d, Hkv, N, B, kTile, ts.kv)) != S2A_OK) return rc;
    if ((rc = make_tmap(&p.tm_o, o, d, H, N, B, kTile)) != S2A_OK) return rc;
    p.o = static_cast<__nv_bfloat16*>(o);
    p.lse = lse;
    p.status = ds->status_ptr;
    p.host_status = ds->host_word_dev;
    p.geo = make_geometry(B, N, H, Hkv, G, n_unshifted, shift, flags);
    p.single = take_single_tiles(p.geo, H, ds->n_sm);
    p.pairs_per_group = most_pairs(p.geo, p.single);
    p.order = BlockOrder(B * H * p.geo.groups, p.pairs_per_group, unit_chunk(static_cast<long long>(G) * d * 2 * 4));  // q, k, v, o
    p.by_heads = FastDiv(H);
    p.scale_log2 = scale * kLog2eHost;
    cudaError_t e = launch_fwd(p, d, static_cast<cudaStream_t>(stream), is_short(p.geo, d, ds->n_sm));
    return e == cudaSuccess ? S2A_OK : cuda_fail(e);
}
}  // namespace

int s2a_fwd_ex(const void* q, const void* k, const void* v, void* o, float* lse, int B, int N, int H, int Hkv, int d,
               int G, float scale, int n_unshifted, int shift, unsigned flags, void* stream) {
    return fwd_impl(q, k, v, o, lse, B, N, H, Hkv, d, G, scale, n_unshifted, shift, flags, stream, TokStrides());
}

int s2a_fwd_packed(const void* qkv, void* o, float* lse, int B, int N, int H, int d, int G, void* stream) {
    if (!qkv) return S2A_ERR_INVALID_ARG;
    if (const int bad = check_default_shape(N, H, d, G)) return bad;
    const __nv_bfloat16* base = static_cast<const __nv_bfloat16*>(qkv);
    const long long hd = static_cast<long long>(H) * d;
    TokStrides ts;
    ts.q = ts.kv = 3 * hd;
    return fwd_impl(base, base + hd, base + 2 * hd, o, lse, B, N, H, H, d, G, 1.0f / sqrtf(static_cast<float>(d)), H / 2,
                    G / 2, 0u, stream, ts);
}

int s2a_fwd(const void* q, const void* k, const void* v, void* o, float* lse, int B, int N, int H, int Hkv, int d,
            int G, void* stream) {
    if (const int bad = check_default_shape(N, H, d, G)) return bad;
    return s2a_fwd_ex(q, k, v, o, lse, B, N, H, Hkv, d, G, 1.0f / sqrtf(static_cast<float>(d)), H / 2, G / 2, 0u, stream);
}

namespace {
// Workspace layout: D [B, H, N] fp32 padded to 256 bytes, 256 reserved bytes (together the minimum; the
// sizes callers were told stay what they were), then the spill area.
constexpr size_t kReservedBytes = 256;
size_t d_bytes(int B, int N, int H) {
    return (static_cast<size_t>(B) * H * N * sizeof(float) + 255) & ~static_cast<size_t>(255);
}
}  // namespace

size_t s2a_bwd_workspace_bytes(int B, int N, int H, int Hkv, int d, int G) {
    if (B <= 0 || N <= 0 || H <= 0 || Hkv <= 0 || d <= 0 || G <= 0) return 0;
    if (N % G != 0 || H % Hkv != 0) return 0;
    return d_bytes(B, N, H) + kReservedBytes;
}

namespace {
constexpr size_t kSpillBlockBytes = static_cast<size_t>(kSpillBlockElems) * 2;
// spill blocks of one KV head with its query heads, for groups of at most T tiles
size_t spill_blocks_per_kv_head(int B, int N, int H, int Hkv, int G, int T) {
    return static_cast<size_t>(B) * (H / Hkv) * (N / G) * static_cast<size_t>(spill_blocks_per_unit(T));
}
}  // namespace

size_t s2a_bwd_workspace_bytes_fast(int B, int N, int H, int Hkv, int d, int G, size_t budget) {
    const size_t min_bytes = s2a_bwd_workspace_bytes(B, N, H, Hkv, d, G);
    if (min_bytes == 0) return 0;
    // tiles of the largest group: G / 128 when G and the default shift G / 2 are multiples of the tile,
    // otherwise one partial tile per run of the group that wraps
    const int T = (G % (2 * kTile) == 0) ? G / kTile : (G + kTile - 1) / kTile + 1;
    const size_t per_kv = spill_blocks_per_kv_head(B, N, H, Hkv, G, T) * kSpillBlockBytes;
    if (budget <= min_bytes) return min_bytes;
    size_t nk = (budget - min_bytes) / per_kv;
    if (nk > static_cast<size_t>(Hkv)) nk = Hkv;
    return nk == 0 ? min_bytes : min_bytes + nk * per_kv;
}

namespace {
enum : unsigned { kStagePre = 1u, kStageDkDv = 2u, kStageDq = 4u, kStageAll = 7u };

int bwd_impl(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* dO, void* dq,
             void* dk, void* dv, int B, int N, int H, int Hkv, int d, int G, float scale, int n_unshifted, int shift,
             void* workspace, size_t workspace_bytes, void* stream, unsigned stages, unsigned flags = 0u,
             const TokStrides& ts = TokStrides(), bool may_spill = true) {
    if (!q || !k || !v || !o || !lse || !dO || !dq || !dk || !dv || !workspace) return S2A_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(o) || !aligned16(lse) || !aligned16(dO) ||
        !aligned16(dq) || !aligned16(dk) || !aligned16(dv))
        return S2A_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return S2A_ERR_INVALID_ARG;
    int rc = check_shape(B, N, H, Hkv, d, G, scale, n_unshifted, shift);
    if (rc != S2A_OK) return rc;
    if (static_cast<long long>(B) * N * H > 0x7fffffffLL) return S2A_ERR_UNSUPPORTED;  // PreParams::rows
    if (workspace_bytes < s2a_bwd_workspace_bytes(B, N, H, Hkv, d, G)) return S2A_ERR_INVALID_ARG;
    DeviceState* ds = nullptr;
    rc = prepare_device(&ds);
    if (rc != S2A_OK) return rc;
    if (*ds->host_word != 0) return S2A_ERR_TIMEOUT;  // an earlier launch gave up: see s2a_device_status()
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!flags_ok(flags)) return S2A_ERR_INVALID_ARG;
    const Geometry geo = make_geometry(B, N, H, Hkv, G, n_unshifted, shift, flags);
    float* Dsum = static_cast<float*>(workspace);

    BwdDkDvParams pk;
    memset(&pk, 0, sizeof pk);
    if ((rc = make_tmap(&pk.tm_k, k, d, Hkv, N, B, kTile, ts.kv)) != S2A_OK) return rc;
    if ((rc = make_tmap(&pk.tm_v, v, d, Hkv, N, B, kTile, ts.kv)) != S2A_OK) return rc;
    if ((rc = make_tmap(&pk.tm_q, q, d, H, N, B, kSubTile, ts.q)) != S2A_OK) return rc;
    if ((rc = make_tmap(&pk.tm_do, dO, d, H, N, B, kSubTile)) != S2A_OK) return rc;
    if ((rc = make_tmap(&pk.tm_dk, dk, d, Hkv, N, B, 32, ts.dkv)) != S2A_OK) return rc;
    if ((rc = make_tmap(&pk.tm_dv, dv, d, Hkv, N, B, 32, ts.dkv)) != S2A_OK) return rc;
    pk.dkv_tok_stride = ts.dkv ? ts.dkv : static_cast<long long>(Hkv) * d;
    pk.lse = lse, pk.Dsum = Dsum;
    pk.dk = static_cast<__nv_bfloat16*>(dk), pk.dv = static_cast<__nv_bfloat16*>(dv);
    pk.status = ds->status_ptr, pk.host_status = ds->host_word_dev, pk.geo = geo, pk.scale = scale, pk.scale_log2 = scale * kLog2eHost;
    pk.spill = nullptr;
    pk.pass.hk0 = 0, pk.pass.nk = Hkv;
    const int chunk_kv = unit_chunk(static_cast<long long>(G) * d * 2 * (2 * (H / Hkv) + 2));  // q and dO of every query head, k, v
    pk.order = BlockOrder(B * Hkv * geo.groups, geo.tiles_per_group, chunk_kv), pk.by_heads = FastDiv(Hkv);

    PreParams pp;
    pp.o = static_cast<const __nv_bfloat16*>(o), pp.dO = static_cast<const __nv_bfloat16*>(dO), pp.Dsum = Dsum;
    pp.rows = B * N * H, pp.N = N, pp.H = H, pp.by_heads = FastDiv(H), pp.by_tokens = FastDiv(N);

    // How many KV heads' worth of dS^T the workspace can hold beyond D: with room for at least one, the
    // dK,dV kernel spills dS^T and dQ is a plain product (several passes over the KV heads if they do
    // not all fit); otherwise dQ recomputes S and dP.  A single-stage call spills only in one pass, so
    // that stages 0, 1, 2 in order stay equal to the whole backward.
    const size_t min_bytes = s2a_bwd_workspace_bytes(B, N, H, Hkv, d, G);
    const size_t per_kv = spill_blocks_per_kv_head(B, N, H, Hkv, G, geo.tiles_per_group);
    size_t nk_fit = 0;
    if (may_spill && workspace_bytes > min_bytes)
        nk_fit = (workspace_bytes - min_bytes) / (per_kv * kSpillBlockBytes);
    if (nk_fit > static_cast<size_t>(Hkv)) nk_fit = Hkv;
    if (stages != kStageAll && nk_fit < static_cast<size_t>(Hkv)) nk_fit = 0;

    const bool overlap = is_short(geo, d, ds->n_sm);
    char* base = static_cast<char*>(workspace);
    cudaError_t e;
    if (stages & kStagePre) {
        e = launch_bwd_preprocess(pp, d, st, overlap);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    if (nk_fit == 0) {
        if (stages & kStageDkDv) {
            e = launch_bwd_dkdv(pk, d, st);
            if (e != cudaSuccess) return cuda_fail(e);
        }
        if (stages & kStageDq) {
            BwdDqParams pq;
            memset(&pq, 0, sizeof pq);
            if ((rc = make_tmap(&pq.tm_q, q, d, H, N, B, kTile, ts.q)) != S2A_OK) return rc;
            if ((rc = make_tmap(&pq.tm_do, dO, d, H, N, B, kTile)) != S2A_OK) return rc;
            pq.tm_k = pk.tm_k, pq.tm_v = pk.tm_v;
            pq.order = BlockOrder(B * H * geo.groups, geo.tiles_per_group, unit_chunk(static_cast<long long>(G) * d * 2 * 4));  // q, dO, k, v
            pq.by_heads = FastDiv(H);
            pq.dq_tok_stride = ts.dq ? ts.dq : static_cast<long long>(H) * d;
            pq.lse = lse, pq.Dsum = Dsum, pq.dq = static_cast<__nv_bfloat16*>(dq);
            pq.status = ds->status_ptr, pq.host_status = ds->host_word_dev, pq.geo = geo, pq.scale = scale, pq.scale_log2 = scale * kLog2eHost;
            e = launch_bwd_dq(pq, d, st, overlap);
            if (e != cudaSuccess) return cuda_fail(e);
        }
        return S2A_OK;
    }

    pk.spill = reinterpret_cast<__nv_bfloat16*>(base + min_bytes);
    BwdDqSpillParams ps;
    memset(&ps, 0, sizeof ps);
    ps.tm_k = pk.tm_k;
    if ((rc = make_tmap(&ps.tm_dq, dq, d, H, N, B, 32, ts.dq)) != S2A_OK) return rc;
    ps.spill = pk.spill;
    ps.dq = static_cast<__nv_bfloat16*>(dq), ps.dq_tok_stride = ts.dq ? ts.dq : static_cast<long long>(H) * d;
    ps.status = ds->status_ptr, ps.host_status = ds->host_word_dev, ps.geo = geo, ps.scale = scale;
    for (int hk0 = 0; hk0 < Hkv; hk0 += static_cast<int>(nk_fit)) {
        const int nk = Hkv - hk0 < static_cast<int>(nk_fit) ? Hkv - hk0 : static_cast<int>(nk_fit);
        pk.pass.hk0 = hk0, pk.pass.nk = nk;
        ps.pass = pk.pass;
        ps.single = take_single_tiles(geo, nk * (H / Hkv), ds->n_sm);
        ps.pairs_per_group = most_pairs(geo, ps.single);
        pk.order = BlockOrder(B * nk * geo.groups, geo.tiles_per_group, chunk_kv), pk.by_heads = FastDiv(nk);
        // what streams through the product kernel, dS, is read once: chunks of 4 to 16 units make no difference
        ps.by_heads = FastDiv(nk * (H / Hkv));
        ps.order = BlockOrder(B * nk * (H / Hkv) * geo.groups, ps.pairs_per_group, kUnitChunk);
        if (stages & kStageDkDv) {
            e = launch_bwd_dkdv(pk, d, st);
            if (e != cudaSuccess) return cuda_fail(e);
        }
        if (stages & kStageDq) {
            e = launch_bwd_dq_spill(ps, d, st, overlap);
            if (e != cudaSuccess) return cuda_fail(e);
        }
    }
    return S2A_OK;
}
}  // namespace

int s2a_bwd_ex(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* dO, void* dq,
               void* dk, void* dv, int B, int N, int H, int Hkv, int d, int G, float scale, int n_unshifted,
               int shift, unsigned flags, void* workspace, size_t workspace_bytes, void* stream) {
    return bwd_impl(q, k, v, o, lse, dO, dq, dk, dv, B, N, H, Hkv, d, G, scale, n_unshifted, shift, workspace,
                    workspace_bytes, stream, kStageAll, flags);
}

int s2a_bwd_packed(const void* qkv, const void* o, const float* lse, const void* dO, void* dqkv, int B, int N, int H,
                   int d, int G, void* workspace, size_t workspace_bytes, void* stream) {
    if (!qkv || !dqkv) return S2A_ERR_INVALID_ARG;
    if (const int bad = check_default_shape(N, H, d, G)) return bad;
    const __nv_bfloat16* in = static_cast<const __nv_bfloat16*>(qkv);
    __nv_bfloat16* out = static_cast<__nv_bfloat16*>(dqkv);
    const long long hd = static_cast<long long>(H) * d;
    TokStrides ts;
    ts.q = ts.kv = ts.dq = ts.dkv = 3 * hd;
    return bwd_impl(in, in + hd, in + 2 * hd, o, lse, dO, out, out + hd, out + 2 * hd, B, N, H, H, d, G,
                    1.0f / sqrtf(static_cast<float>(d)), H / 2, G / 2, workspace, workspace_bytes, stream, kStageAll, 0u, ts);
}

int s2a_bwd_stage(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* dO,
                  void* dq, void* dk, void* dv, int B, int N, int H, int Hkv, int d, int G, void* workspace,
                  size_t workspace_bytes, int stage, void* stream) {
    if (stage < 0 || stage > 2) return S2A_ERR_INVALID_ARG;
    if (const int bad = check_default_shape(N, H, d, G)) return bad;
    return bwd_impl(q, k, v, o, lse, dO, dq, dk, dv, B, N, H, Hkv, d, G, 1.0f / sqrtf(static_cast<float>(d)), H / 2,
                    G / 2, workspace, workspace_bytes, stream, 1u << stage);
}

int s2a_bwd(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* dO, void* dq,
            void* dk, void* dv, int B, int N, int H, int Hkv, int d, int G, void* workspace, size_t workspace_bytes,
            void* stream) {
    if (const int bad = check_default_shape(N, H, d, G)) return bad;
    return s2a_bwd_ex(q, k, v, o, lse, dO, dq, dk, dv, B, N, H, Hkv, d, G, 1.0f / sqrtf(static_cast<float>(d)), H / 2,
                      G / 2, 0u, workspace, workspace_bytes, stream);
}

int s2a_fwd_bwd_host(const void* h_q, const void* h_k, const void* h_v, const void* h_dO, void* h_o, float* h_lse,
                     void* h_dq, void* h_dk, void* h_dv, void* d_q, void* d_k, void* d_v, void* d_dO, void* d_o,
                     float* d_lse, void* d_dq, void* d_dk, void* d_dv, int B, int N, int H, int Hkv, int d, int G,
                     void* workspace, size_t workspace_bytes, void* stream) {
    if (!h_q || !h_k || !h_v || !h_dO || !h_o || !h_lse || !h_dq || !h_dk || !h_dv) return S2A_ERR_INVALID_ARG;
    if (!d_q || !d_k || !d_v || !d_dO || !d_o || !d_lse || !d_dq || !d_dk || !d_dv) return S2A_ERR_INVALID_ARG;
    if (const int bad = check_default_shape(N, H, d, G)) return bad;
    int rc = check_shape(B, N, H, Hkv, d, G, 1.0f, H / 2, G / 2);
    if (rc != S2A_OK) return rc;
    // a refusal comes before the first copy is enqueued, so what the kernels' launchers ask is asked here as well
    const void* const buffers[] = {d_q, d_k, d_v, d_dO, d_o, d_lse, d_dq, d_dk, d_dv};
    for (const void* p : buffers)
        if (!aligned16(p)) return S2A_ERR_INVALID_ARG;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return S2A_ERR_INVALID_ARG;
    if (workspace_bytes < s2a_bwd_workspace_bytes(B, N, H, Hkv, d, G)) return S2A_ERR_INVALID_ARG;
    DeviceState* ds = nullptr;
    if ((rc = prepare_device(&ds)) != S2A_OK) return rc;
    if (*ds->host_word != 0) return S2A_ERR_TIMEOUT;  // an earlier launch gave up: see s2a_device_status()
    cudaError_t e;
    std::lock_guard<std::mutex> lock(ds->host_path);
    if (!ds->host_path_ready) {
        if ((e = cudaStreamCreateWithFlags(&ds->copy_in, cudaStreamNonBlocking)) != cudaSuccess) return cuda_fail(e);
        if ((e = cudaStreamCreateWithFlags(&ds->copy_out, cudaStreamNonBlocking)) != cudaSuccess) return cuda_fail(e);
        for (cudaEvent_t* ev : {&ds->ev_start, &ds->ev_done, &ds->ev_in_done, &ds->ev_qkv, &ds->ev_do, &ds->ev_fwd, &ds->ev_bwd})
            if ((e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming)) != cudaSuccess) return cuda_fail(e);
        ds->host_path_ready = true;
    }
    // Heads and groups are independent, so the job is cut into chunks (host_plan.h): while chunk c is
    // computed, chunk c + 1 travels to the device and the results of chunk c - 1 travel back.  The forward
    // pass of a chunk runs while its dO is on its way, and o goes back while its backward pass runs.
    const int rep = H / Hkv;
    const size_t hb = static_cast<size_t>(d) * 2;  // bytes of one head of one token
    const float scale = 1.0f / sqrtf(static_cast<float>(d));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    auto at = [](const void* base, size_t bytes) { return const_cast<char*>(static_cast<const char*>(base)) + bytes; };

    if ((e = cudaEventRecord(ds->ev_start, st)) != cudaSuccess) return cuda_fail(e);
    // From here on work may sit in the two copy streams: whatever happens, `stream` is made to wait
    // for both before this function returns, so that the caller's synchronisation covers it all.
    auto join = [&]() -> cudaError_t {
        cudaError_t e1 = cudaEventRecord(ds->ev_done, ds->copy_out);
        if (e1 == cudaSuccess) e1 = cudaStreamWaitEvent(st, ds->ev_done, 0);
        cudaError_t e2 = cudaEventRecord(ds->ev_in_done, ds->copy_in);
        if (e2 == cudaSuccess) e2 = cudaStreamWaitEvent(st, ds->ev_in_done, 0);
        return e1 != cudaSuccess ? e1 : e2;
    };
    auto enqueue_all = [&]() -> int {
        if ((e = cudaStreamWaitEvent(ds->copy_in, ds->ev_start, 0)) != cudaSuccess) return cuda_fail(e);
        if ((e = cudaStreamWaitEvent(ds->copy_out, ds->ev_start, 0)) != cudaSuccess) return cuda_fail(e);
        size_t at_q = 0, at_kv = 0;  // (token, head) rows of the chunks before this one
        return cut_host_job(B, N, H, Hkv, d, G, [&](const HostChunk& c) -> int {
            const int n = c.tokens(), hc = c.kvn * rep, h0 = c.kv0 * rep;
            void *cq = at(d_q, at_q * hb), *ck = at(d_k, at_kv * hb), *cv = at(d_v, at_kv * hb), *cdo = at(d_dO, at_q * hb);
            void *co = at(d_o, at_q * hb), *cdq = at(d_dq, at_q * hb), *cdk = at(d_dk, at_kv * hb), *cdv = at(d_dv, at_kv * hb);
            float* cl = d_lse + at_q;
            at_q += static_cast<size_t>(c.bn) * n * hc, at_kv += static_cast<size_t>(c.bn) * n * c.kvn;
            // `heads` heads from `first` on, of a tensor with `all` heads, for the chunk's tokens; several batch items come with all N
            auto copy = [&](cudaMemcpyKind kind, const void* host, void* dev, int all, int first, int heads) -> cudaError_t {
                const size_t w = heads * hb, pitch = all * hb;
                size_t row = 0;
                for (int r = 0; r < 2; ++r) {
                    if (c.n[r] == 0) continue;
                    void* h = at(host, (static_cast<size_t>(c.b0) * N + c.from[r]) * pitch + first * hb);
                    void* g = at(dev, row * w);
                    const size_t rows = static_cast<size_t>(c.bn) * c.n[r];
                    const cudaError_t ec = kind == cudaMemcpyHostToDevice
                                               ? cudaMemcpy2DAsync(g, w, h, pitch, w, rows, kind, ds->copy_in)
                                               : cudaMemcpy2DAsync(h, pitch, g, w, w, rows, kind, ds->copy_out);
                    if (ec != cudaSuccess) return ec;
                    row += rows;
                }
                return cudaSuccess;
            };
            auto copy_lse = [&]() -> cudaError_t {
                float* h = h_lse + (static_cast<size_t>(c.b0) * H + h0) * N;
                const size_t f = sizeof(float);
                if (n == N) return cudaMemcpy2DAsync(h, H * f * N, cl, hc * f * N, hc * f * N, c.bn, cudaMemcpyDeviceToHost, ds->copy_out);
                for (int r = 0, row = 0; r < 2; row += c.n[r], ++r) {
                    if (c.n[r] == 0) continue;
                    const cudaError_t ec = cudaMemcpy2DAsync(h + c.from[r], f * N, cl + row, f * n, f * c.n[r], hc, cudaMemcpyDeviceToHost, ds->copy_out);
                    if (ec != cudaSuccess) return ec;
                }
                return cudaSuccess;
            };
            auto after = [](cudaStream_t waiting, cudaEvent_t ev, cudaStream_t done) -> cudaError_t {
                const cudaError_t ec = cudaEventRecord(ev, done);
                return ec != cudaSuccess ? ec : cudaStreamWaitEvent(waiting, ev, 0);
            };
            // host -> device, and the forward pass behind q, k, v
            if ((e = copy(cudaMemcpyHostToDevice, h_q, cq, H, h0, hc)) != cudaSuccess) return cuda_fail(e);
            if ((e = copy(cudaMemcpyHostToDevice, h_k, ck, Hkv, c.kv0, c.kvn)) != cudaSuccess) return cuda_fail(e);
            if ((e = copy(cudaMemcpyHostToDevice, h_v, cv, Hkv, c.kv0, c.kvn)) != cudaSuccess) return cuda_fail(e);
            if ((e = after(st, ds->ev_qkv, ds->copy_in)) != cudaSuccess) return cuda_fail(e);
            if ((e = copy(cudaMemcpyHostToDevice, h_dO, cdo, H, h0, hc)) != cudaSuccess) return cuda_fail(e);
            int rc2 = fwd_impl(cq, ck, cv, co, cl, c.bn, n, hc, c.kvn, d, G, scale, c.n_unshifted, c.shift, 0u, stream, TokStrides());
            if (rc2 != S2A_OK) return rc2;
            // o and lse go back while the backward pass runs behind dO
            if ((e = after(ds->copy_out, ds->ev_fwd, st)) != cudaSuccess) return cuda_fail(e);
            if ((e = copy(cudaMemcpyDeviceToHost, h_o, co, H, h0, hc)) != cudaSuccess) return cuda_fail(e);
            if ((e = copy_lse()) != cudaSuccess) return cuda_fail(e);
            if ((e = after(st, ds->ev_do, ds->copy_in)) != cudaSuccess) return cuda_fail(e);
            rc2 = bwd_impl(cq, ck, cv, co, cl, cdo, cdq, cdk, cdv, c.bn, n, hc, c.kvn, d, G, scale, c.n_unshifted, c.shift, workspace,
                           workspace_bytes, stream, kStageAll);
            if (rc2 != S2A_OK) return rc2;
            if ((e = after(ds->copy_out, ds->ev_bwd, st)) != cudaSuccess) return cuda_fail(e);
            if ((e = copy(cudaMemcpyDeviceToHost, h_dq, cdq, H, h0, hc)) != cudaSuccess) return cuda_fail(e);
            if ((e = copy(cudaMemcpyDeviceToHost, h_dk, cdk, Hkv, c.kv0, c.kvn)) != cudaSuccess) return cuda_fail(e);
            if ((e = copy(cudaMemcpyDeviceToHost, h_dv, cdv, Hkv, c.kv0, c.kvn)) != cudaSuccess) return cuda_fail(e);
            return S2A_OK;
        });
    };
    rc = enqueue_all();
    // the caller's stream is done when the last copy back is (also after a failure part-way)
    const int saved_cuda_error = tl_last_cuda_error;
    const cudaError_t ej = join();
    if (rc != S2A_OK) {
        tl_last_cuda_error = saved_cuda_error;
        return rc;
    }
    return ej == cudaSuccess ? S2A_OK : cuda_fail(ej);
}

// ---------------------------------------------------------------------------------------------
// Backward without caller-provided scratch
// ---------------------------------------------------------------------------------------------
namespace {

// Built-in home for D = rowsum(dO * o) when the caller cannot provide a workspace: 2^20 fp32 rows and
// the reserved bytes of a workspace (4 MiB in all), which every GPU that loads this library keeps
// resident until the process exits.
constexpr size_t kBuiltinScratchRows = size_t(1) << 20;
static __device__ __align__(256) float g_builtin_scratch[kBuiltinScratchRows + kReservedBytes / sizeof(float)];

// In host code `g_builtin_scratch` is only a handle for the runtime, not an address a kernel may
// use; the device address is looked up once per device, with that device current.
float* g_builtin_scratch_ptr[kMaxDevices] = {};

int builtin_scratch(float** out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e);
    if (dev < 0 || dev >= kMaxDevices) return S2A_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_dev_mutex);
    if (!g_builtin_scratch_ptr[dev]) {
        void* ptr = nullptr;
        e = cudaGetSymbolAddress(&ptr, g_builtin_scratch);
        if (e != cudaSuccess) return cuda_fail(e);
        g_builtin_scratch_ptr[dev] = static_cast<float*>(ptr);
    }
    *out = g_builtin_scratch_ptr[dev];
    return S2A_OK;
}

}  // namespace

int s2a_bwd_noalloc(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* dO,
                    void* dq, void* dk, void* dv, int B, int N, int H, int Hkv, int d, int G, void* stream) {
    if (B <= 0 || N <= 0 || H <= 0) return S2A_ERR_INVALID_ARG;
    if (static_cast<unsigned long long>(B) * static_cast<unsigned long long>(H) * static_cast<unsigned long long>(N) >
        kBuiltinScratchRows)
        return S2A_ERR_TOO_LARGE;
    if (const int bad = check_default_shape(N, H, d, G)) return bad;
    float* scratch = nullptr;
    const int rc = builtin_scratch(&scratch);
    if (rc != S2A_OK) return rc;
    // Every row of D that the two gradient kernels read is rewritten by the first kernel of this
    // call, so nothing left in the array by an earlier call matters.
    return bwd_impl(q, k, v, o, lse, dO, dq, dk, dv, B, N, H, Hkv, d, G, 1.0f / sqrtf(static_cast<float>(d)), H / 2,
                    G / 2, scratch, kBuiltinScratchRows * sizeof(float) + kReservedBytes, stream, kStageAll, 0u, TokStrides(), false);
}

size_t s2a_bwd_noalloc_max_rows(void) { return kBuiltinScratchRows; }

int s2a_selftest_wait_expiry(long long limit_cycles, void* stream) {
    if (limit_cycles < 1 || limit_cycles > kWaitLimitCycles) return S2A_ERR_INVALID_ARG;
    DeviceState* ds = nullptr;
    const int rc = prepare_device(&ds);
    if (rc != S2A_OK) return rc;
    s2a_wait_selftest_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(ds->status_ptr, ds->host_word_dev, limit_cycles);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? S2A_OK : cuda_fail(e);
}

int s2a_device_status(int* where) {
    DeviceState* ds = nullptr;
    int rc = prepare_device(&ds);
    if (rc != S2A_OK) return rc;
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return cuda_fail(e);
    int word = 0;
    e = cudaMemcpy(&word, ds->status_ptr, sizeof word, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e);
    if (word != 0) {
        const int zero = 0;
        e = cudaMemcpy(ds->status_ptr, &zero, sizeof zero, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return cuda_fail(e);
        *ds->host_word = 0;
        if (where) *where = word;
        return S2A_ERR_TIMEOUT;
    }
    if (where) *where = 0;
    return S2A_OK;
}

}  // extern "C"
#pragma GCC visibility pop
