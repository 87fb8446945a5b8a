// Kernel parameter blocks and launcher declarations shared by the host entry points and the kernels.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace s2a {

constexpr int kTile = 128;     // tokens per resident tile (query rows in forward / dQ, key rows in dK,dV)
constexpr int kSubTile = 64;   // tokens per streamed tile in the backward kernels

// Codes recorded when a bounded device-side wait expires: kernel id * 100 + wait id.
enum WaitCode : int {
    kWaitFwd = 100,
    kWaitBwdDq = 200,
    kWaitBwdDkDv = 300,
    kWaitBwdDqSpill = 400,
};

// Block order shared by the tensor-core kernels.  A "unit" is one (batch, head, group); it has
// `tiles` tiles whose cost falls with their rank (rank 0 = most work).  Units are taken in chunks:
// inside a chunk all rank-0 tiles come first, then all rank-1 tiles, and so on.  So the
// blocks that run together belong to a few units (their streamed operands stay in L2), heavy tiles
// start first, and the tail of the grid consists of the lightest tiles only.
constexpr int kUnitChunk = 8;
// Units in a chunk where their operands are what the L2 is for (`unit_bytes` each): as many as keep them
// within a quarter of it, rounded down to a power of two (most counts of units divide by it), at least two.
// A chunk's first tiles are its heavy ones, and those of the last chunk start when the launch is nearly over:
// the more units it has, the more light tiles are left to even out the ends.  Measured with chunks of 8 and of
// this rule: dK,dV 153 and 138 us on 4 x 2048 tokens with groups of 512 (64 units), 138 and 127 on a grouped-query
// shape (16 units).  Chunks that overflow the L2 cost more than the ends: 32k, units of 8 MB, forward 1.98 ms
// with 3, 1.99 with 8, 2.10 with 24; 100k, units of 26 MB, 17.4 ms with 2, 18.1 with 8, 20.6 with 64.
constexpr long long kChunkBytes = 32ll << 20;
__host__ __device__ inline int unit_chunk(long long unit_bytes) {
    int n = 2;
    while (n < 4096 && 2 * n * unit_bytes <= kChunkBytes) n *= 2;
    return n;
}
// n / d for 0 <= n < 2^31 as a multiplication (d, and with it the multiplier, is known when the kernel is
// launched): decoding a work item takes about seven divisions one after the other, on one thread, while the
// other warps wait for the item.  dK,dV kernel, division and multiplication, us a launch in a loop: Llama2-7B 16k 951
// and 909, 8k 275 and 264, 4 x 2048 tokens with groups of 512 120 and 113.
struct FastDiv {
    uint32_t d = 1, m = 0;
    int s = 0;
    FastDiv() = default;
    explicit FastDiv(int divisor) : d(static_cast<uint32_t>(divisor)) {
        if (divisor <= 1) return;
        int l = 1;  // 2^(l-1) < d <= 2^l
        while ((1ull << l) < d) ++l;
        m = static_cast<uint32_t>(((1ull << (31 + l)) + d - 1) / d);  // n m / 2^(31+l) is exact for n < 2^31
        s = l - 1;
    }
    __host__ __device__ int operator()(int n) const {
        if (d <= 1) return n;
#ifdef __CUDA_ARCH__
        return static_cast<int>(__umulhi(static_cast<uint32_t>(n), m) >> s);
#else
        return static_cast<int>((static_cast<uint64_t>(static_cast<uint32_t>(n)) * m) >> 32 >> s);
#endif
    }
    // n / d; *rest = n % d
    __host__ __device__ int operator()(int n, int* rest) const {
        const int q = (*this)(n);
        *rest = n - q * static_cast<int>(d);
        return q;
    }
};

// The block order of a launch: `units` units of `tiles` tiles in chunks of `chunk` units.
struct BlockOrder {
    int units = 0, chunk = 1, tail = 0;  // tail: first unit of the last chunk, which can be smaller
    FastDiv per_chunk, in_chunk, in_tail;
    BlockOrder() = default;
    BlockOrder(int units_, int tiles, int chunk_) : units(units_), chunk(chunk_ < units_ ? chunk_ : units_) {
        tail = (units - 1) / chunk * chunk;
        per_chunk = FastDiv(chunk * tiles), in_chunk = FastDiv(chunk), in_tail = FastDiv(units - tail);
    }
    __host__ __device__ void decode(int idx, int* unit, int* rank) const {
        int within, at;
        const int first = per_chunk(idx, &within) * chunk;
        *rank = first == tail ? in_tail(within, &at) : in_chunk(within, &at);
        *unit = first + at;
    }
};
inline void decode_block(long long idx, int units, int tiles, int* unit, int* rank, int unit_chunk = kUnitChunk) {
    BlockOrder(units, tiles, unit_chunk).decode(static_cast<int>(idx), unit, rank);
}

// Geometry of the shifted grouping (Algorithm 1): common to every kernel.
struct Geometry {
    int B, N, H, Hkv, G;
    int n_unshifted;      // heads [0, n_unshifted) use the unshifted partition
    int shift;            // tokens; the rest of the heads are rolled by -shift (G/2 in Algorithm 1)
    int tiles_per_group;  // largest number of 128-token tiles any group has (G / 128 when G and shift are multiples of 128)
    int groups;           // N / G
    int leak_free;        // variant 2 of Appendix B: cut the wrapped group of a shifted head at the wrap
    int swap_wrapped;     // variant 3 of Appendix B: the two runs of the wrapped group change places
    int rep;              // query heads of a KV head, H / Hkv
    FastDiv by_group, by_groups, by_rep;  // divisions by G, by groups and by rep
};

// Where the tokens of one group live.  Group g of a head with shift s holds rolled positions
// [g G, (g+1) G), i.e. original tokens (x + s) mod N: one run [a0, a0 + lenA) and, only in the group
// that wraps past token N-1, a second run [0, lenB).  Each run is cut into 128-token tiles from its own
// start, so a tile is always a contiguous range of original tokens (one TMA box, no wrap inside a
// tile) and only the last tile of a run can have fewer than 128 valid rows.  Tiles are numbered in
// causal order: the nA tiles of the first run, then those of the second (the other way round in
// variant 3 of Appendix B).
struct GroupLayout {
    int a0, lenA, lenB;
    int nA, nTiles;
    int cut;      // variant 2: tile index at which the wrapped group is cut in two (0 = no cut)
    int swapped;  // variant 3: the tiles of the second run ([0, lenB), the front of the sequence) come first
};
__host__ __device__ inline GroupLayout group_layout(const Geometry& geo, int s, int g) {
    GroupLayout L;
    int a = g * geo.G + s;  // in (-N, 2 N), and 2 N < 2^31
    if (a < 0) a += geo.N;
    if (a >= geo.N) a -= geo.N;
    L.a0 = a;
    L.lenA = (geo.N - L.a0 < geo.G) ? geo.N - L.a0 : geo.G;
    L.lenB = geo.G - L.lenA;
    L.nA = (L.lenA + kTile - 1) / kTile;
    L.nTiles = L.nA + (L.lenB + kTile - 1) / kTile;
    // Variant 2: the second run starts at original token 0; queries there attend keys from the cut
    // on, keys before the cut are attended by queries before the cut only.
    L.cut = (geo.leak_free && L.lenB > 0) ? L.nA : 0;
    // Variant 3: the wrapped group is attended in original token order, front tokens first.
    L.swapped = (geo.swap_wrapped && L.lenB > 0) ? 1 : 0;
    return L;
}
struct TileRef {
    int tok0;   // original token of row 0
    int valid;  // rows that belong to the group (the rest of the box is other tokens or zero fill)
};
__host__ __device__ inline TileRef tile_ref(const GroupLayout& L, int i) {
    TileRef t;
    const int nFirst = L.swapped ? L.nTiles - L.nA : L.nA;  // tiles of the run that comes first
    const bool in_run_a = L.swapped ? (i >= nFirst) : (i < nFirst);
    const int k = (i < nFirst) ? i : i - nFirst;             // tile within its run
    if (in_run_a) {
        t.tok0 = L.a0 + k * kTile;
        t.valid = L.lenA - k * kTile;
    } else {
        t.tok0 = k * kTile;
        t.valid = L.lenB - k * kTile;
    }
    if (t.valid > kTile) t.valid = kTile;
    return t;
}
// 64-row halves of the tiles, numbered 2 i and 2 i + 1; a half can be empty (valid = 0).
__host__ __device__ inline TileRef subtile_ref(const GroupLayout& L, int n) {
    TileRef t = tile_ref(L, n >> 1);
    const int off = (n & 1) * kSubTile;
    t.tok0 += off;
    t.valid -= off;
    if (t.valid > kSubTile) t.valid = kSubTile;
    if (t.valid < 0) t.valid = 0;
    return t;
}
// Causal range in tiles: query tile i attends key tiles [first_key_tile, i]; key tile j is attended
// by query tiles [j, end_query_tile).
__host__ __device__ inline int first_key_tile(const GroupLayout& L, int i) { return (L.cut > 0 && i >= L.cut) ? L.cut : 0; }
__host__ __device__ inline int end_query_tile(const GroupLayout& L, int j) { return (L.cut > 0 && j < L.cut) ? L.cut : L.nTiles; }

// The forward kernel and the dQ product kernel work on two neighbouring query tiles of a group at a time
// ("a pair"), which share the key tiles they stream.  The pairs of a group are numbered by rank, most work first; the tiles on
// either side of a cut (variant 2 of Appendix B) have no keys in common and are paired separately.  Where
// a problem has fewer pairs than the GPU has multiprocessors the kernels take single tiles instead
// (`single`; a pair of which only the second tile exists).
__host__ __device__ inline int pairs_of_group(const GroupLayout& L, bool single = false) {
    if (single) return L.nTiles;
    return L.cut > 0 ? (L.nTiles - L.cut + 1) / 2 + (L.cut + 1) / 2 : (L.nTiles + 1) / 2;
}
struct TilePair {
    int i[2];     // query tiles (i[0] = i[1] - 1)
    int j_begin;  // first key tile; tile t attends key tiles [j_begin, i[t]]
    int n[2];     // key tiles each attends: n[1] = n[0] + 1, n[0] = 0 when there is no second tile
};
__host__ __device__ inline TilePair tile_pair(const GroupLayout& L, int rank, bool single = false) {
    if (single) {
        TilePair t;
        t.i[1] = L.nTiles - 1 - rank;
        t.i[0] = t.i[1] - 1;
        t.j_begin = first_key_tile(L, t.i[1]);
        t.n[1] = t.i[1] + 1 - t.j_begin;
        t.n[0] = 0;
        return t;
    }
    int lo = 0, hi = L.nTiles;  // tiles [lo, hi) hold this pair
    if (L.cut > 0) {
        const int upper = (L.nTiles - L.cut + 1) / 2;
        if (rank < upper) lo = L.cut;
        else hi = L.cut, rank -= upper;
    }
    TilePair t;
    t.j_begin = lo;
    t.i[1] = hi - 1 - 2 * rank;
    t.i[0] = t.i[1] - 1;
    t.n[1] = t.i[1] + 1 - lo;
    t.n[0] = t.i[0] + 1 - lo;  // 0 when i[1] is the first tile of its range
    return t;
}

struct alignas(64) FwdParams {
    CUtensorMap tm_q;  // bf16 (d, H,   N, B), box (64, 1, 128, 1), 128-byte swizzle
    CUtensorMap tm_k;  // bf16 (Hkv * d, 2 tokens apart by two, 2 by one, N / 4, B), box (64, 2, 2, 32, 1): see key_of_column()
    CUtensorMap tm_v;  // bf16 (d, Hkv, N, B), box as tm_q
    CUtensorMap tm_o;  // like tm_q, for the stores of whole tiles
    __nv_bfloat16* o;
    float* lse;
    int* status;       // device status word (see WaitCtx)
    int* host_status;  // its mirror in mapped host memory
    Geometry geo;
    int pairs_per_group;  // largest number of query tile pairs any group has
    bool single;          // work items are single tiles (see tile_pair)
    BlockOrder order;     // of the pairs of (batch, head, group)
    FastDiv by_heads;     // division by H
    float scale_log2;     // softmax scale * log2(e)
};

struct PreParams {
    const __nv_bfloat16* o;
    const __nv_bfloat16* dO;
    float* Dsum;  // [B, H, N]
    int rows;     // B N H; the entry points refuse 2^31 and more (q alone would be 275 GB)
    int N, H;
    FastDiv by_heads, by_tokens;
};

struct alignas(64) BwdDqParams {
    CUtensorMap tm_q, tm_do;  // box (64, 1, 128, 1): the resident query tile
    CUtensorMap tm_k, tm_v;   // box (64, 1, 128, 1): streamed key tiles
    const float* lse;         // [B, H, N]
    const float* Dsum;        // [B, H, N]
    __nv_bfloat16* dq;
    long long dq_tok_stride;  // elements between consecutive tokens of dq (H * d when dense)
    BlockOrder order;         // of the query tiles of (batch, head, group)
    FastDiv by_heads;         // division by H
    int* status;       // device status word (see WaitCtx)
    int* host_status;  // its mirror in mapped host memory
    Geometry geo;
    float scale, scale_log2;
};

// The dK,dV kernel can leave its dS^T values (bf16) in global memory for a dQ kernel that then only
// has to multiply them with K instead of recomputing S and dP.  One pass covers the KV heads
// [hk0, hk0 + nk) with their query heads; a "spill unit" is one (batch, query head of the pass, group),
// numbered (b * nk * rep + (hq - hk0 * rep)) * groups + g.  A unit owns T (T + 1) blocks, T =
// tiles_per_group: block (j, n) holds dS^T of key tile j and 64-query sub-tile n >= 2 j, 128 key rows of
// 64 bf16 (16 KB), stored chunk-major: the 16-byte chunk c (queries 8 c .. 8 c + 7) of key row r sits at
// byte (c * 128 + r) * 16 of the block, which is both what a warp of the dK,dV kernel writes in one
// coalesced store and an operand layout the tensor core reads directly.  Masked entries and rows that
// are not part of the group are zero.
struct SpillPass {
    int hk0, nk;  // KV heads of this pass
};
__host__ __device__ inline long long spill_blocks_per_unit(int T) { return static_cast<long long>(T) * (T + 1); }
__host__ __device__ inline long long spill_block(long long unit, int T, int j, int n) {
    return unit * spill_blocks_per_unit(T) + static_cast<long long>(j) * (2 * T - j + 1) + (n - 2 * j);
}
constexpr int kSpillBlockElems = kTile * kSubTile;  // bf16 values per block

struct alignas(64) BwdDkDvParams {
    CUtensorMap tm_k, tm_v;   // box (64, 1, 128, 1): the resident key tile
    CUtensorMap tm_q, tm_do;  // box (64, 1,  64, 1): streamed query sub-tiles
    CUtensorMap tm_dk, tm_dv; // box (64, 1,  32, 1): stores, 32 key rows at a time
    const float* lse;
    const float* Dsum;
    __nv_bfloat16* dk;
    __nv_bfloat16* dv;
    long long dkv_tok_stride;  // elements between consecutive tokens of dk and dv (Hkv * d when dense)
    __nv_bfloat16* spill;      // dS^T blocks of this pass (spilling variant only)
    SpillPass pass;            // KV heads this launch covers (all of them when nothing is spilled)
    BlockOrder order;          // of the key tiles of (batch, KV head of the pass, group)
    FastDiv by_heads;          // division by the KV heads of the pass
    int* status;       // device status word (see WaitCtx)
    int* host_status;  // its mirror in mapped host memory
    Geometry geo;
    float scale, scale_log2;
};

// dQ from spilled dS^T: dQ_i = scale * sum_j dS_ij K_j, two neighbouring query tiles at a time.
struct alignas(64) BwdDqSpillParams {
    CUtensorMap tm_k;   // box (64, 1, 128, 1): streamed key tiles
    CUtensorMap tm_dq;  // box (64, 1,  32, 1): stores, 32 query rows at a time
    const __nv_bfloat16* spill;  // the blocks the dK,dV kernel of this pass wrote
    __nv_bfloat16* dq;
    long long dq_tok_stride;
    SpillPass pass;
    int* status;
    int* host_status;
    Geometry geo;
    int pairs_per_group;  // largest number of query tile pairs any group has
    bool single;          // work items are single tiles (see tile_pair)
    BlockOrder order;     // of the pairs of (batch, query head of the pass, group)
    FastDiv by_heads;     // division by the query heads of the pass
    float scale;
};

// With `overlap`, programmatic stream serialisation: the kernel's blocks may be set up (barriers, tensor memory,
// descriptors) while the kernel before it in the stream runs its last blocks; see wait_for_predecessor().  The
// entry points ask for it where a launch is short: a forward and a backward of 1024 tokens, 4 heads take 25.6 instead
// of 31.7 us, of 4 x 2000 tokens in groups of 200 96 instead of 102, of 2 x 4096 tokens (grouped query) 275 instead
// of 278.  On larger problems nothing is gained (Llama2-7B 8k: 647 against 629).  The dK,dV kernel is always
// launched plainly: with the two instructions in it it was 2 to 3 % slower from 4 x 2048 tokens upwards.
template <typename Params>
cudaError_t launch_kernel(void (*kernel)(Params), unsigned grid, int threads, int smem_bytes, cudaStream_t stream, const Params& p, bool overlap) {
    cudaLaunchConfig_t config = {};
    config.gridDim = dim3(grid);
    config.blockDim = dim3(static_cast<unsigned>(threads));
    config.dynamicSmemBytes = static_cast<size_t>(smem_bytes);
    config.stream = stream;
    cudaLaunchAttribute attribute = {};
    attribute.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attribute.val.programmaticStreamSerializationAllowed = 1;
    config.attrs = &attribute;
    config.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&config, kernel, p);
}

// Enqueue one kernel each on `stream`; return the launch error, if any.
cudaError_t launch_fwd(const FwdParams& p, int d, cudaStream_t stream, bool overlap);
cudaError_t launch_bwd_preprocess(const PreParams& p, int d, cudaStream_t stream, bool overlap);
cudaError_t launch_bwd_dq(const BwdDqParams& p, int d, cudaStream_t stream, bool overlap);
cudaError_t launch_bwd_dkdv(const BwdDkDvParams& p, int d, cudaStream_t stream);  // p.spill != nullptr: spilling variant
cudaError_t launch_bwd_dq_spill(const BwdDqSpillParams& p, int d, cudaStream_t stream, bool overlap);

// Per-device kernel attribute set-up (dynamic shared memory sizes).
cudaError_t configure_fwd();
cudaError_t configure_bwd();

}  // namespace s2a
