// How s2a_fwd_bwd_host cuts a job into chunks (host code, no CUDA).
#pragma once

namespace s2a {

// One chunk: whole KV heads with their query heads, of some batch items, in the tokens of some groups.  Its rows
// lie in the device buffers as [bn][tok[0] then tok[1] tokens][heads][d], where it is a job of its own: its
// last group wraps around its own end if `shift` is not zero (only the chunk with a shifted head's wrapping group
// has that, and it holds the tokens of both ends in the order of the sequence, so every tile is cut as in the whole job).
struct HostChunk {
    int b0, bn;          // batch items
    int kv0, kvn;        // KV heads
    int from[2], n[2];   // up to two runs of tokens
    int n_unshifted;     // query heads of the chunk whose groups are not shifted
    int shift;
    int tokens() const { return n[0] + n[1]; }
};

// What the call takes is one direction of the link for the whole job, plus the largest chunk (the copies back
// run behind the copies in by one chunk, and a chunk that grows leaves them idle), plus what every chunk costs
// on top of its bytes: 6 us for each of its four or five copies in a direction.  So the chunks are equal, and their
// number balances the last two: sqrt(bytes in / kHostChunkCost), where kHostChunkCost is what the link moves in
// the time of a chunk's copies, 40 us.  Rows stay wide: with both directions busy the copy engines moved 49.9 GB/s
// each way with rows of 4096 bytes, 49.4 at 2048, 46.9 at 1024, 44.9 at 512 and 35.2 at 256.  Batch items are
// cut first (rows of all heads), then the unshifted from the shifted heads and groups of tokens (rows of half
// the heads), then heads while a row of the keys keeps kHostRowBytes, each as long as that brings the number nearer to
// the one wanted and not more than one above it.  More than 16 chunks were slower (32 heads of 128, 32k tokens, groups of
// 8k: 28.2 ms with 32 chunks, 23.9 with 16), and most of all where the cut leaves a narrow chunk for one KV head between the
// halves: 6 x 8192 tokens of 10 heads on 5 10.46 ms with 30 chunks, 9.88 with 18, 9.41 with 6; 13 x 8192 21.1 with 39, 19.6
// with 13; 7 x 4096 tokens of 32 heads 22.2 with 28, 21.5 with 14 (but 12 x 2048 tokens 17.96 with 24, 18.29 with 12).
// Against chunks of 2, 2, 4, 8, 8, 4, 2, 2 of 32 heads for all tokens: that shape 27.9 -> 24.0 ms, 8k tokens 7.20 -> 6.49
// (link: 5.4), 64 heads on 8 at 8k 8.15 -> 7.33, 4 x 2000 tokens of 16 heads on 4 of 64 1.45 -> 1.32, 1k of 4 heads
// of 64, one chunk, 0.207 -> 0.133.
constexpr int kHostChunks = 16;
constexpr long long kHostChunkCost = 2 << 20;
constexpr long long kHostRowBytes = 1024;

// Calls emit(const HostChunk&) for every chunk; a result other than 0 ends it and is returned.
template <typename Emit>
int cut_host_job(int B, int N, int H, int Hkv, int d, int G, Emit&& emit) {
    const int rep = H / Hkv, groups = N / G;
    const long long bytes_in = 4LL * B * N * d * (H + Hkv);
    int want = 1;
    while (want < kHostChunks && (want + 1) * (want + 1) * kHostChunkCost <= bytes_in) ++want;
    const int batches = B < want ? B : want;
    // KV heads [0, half) have unshifted query heads only, [Hkv - half, Hkv) shifted ones only; one between has both
    const int half = H / 2 / rep;
    const int between = Hkv > 2 * half ? 1 : 0;
    // whether either half of the heads of a batch item is rather cut into `parts` parts than into `than` (0: the item stays whole)
    auto nearer = [&](int parts, int than) {
        auto off = [&](int n) {
            const int chunks = batches * (n == 0 ? 1 : 2 * n + between);
            return chunks > want ? chunks - want : want - chunks;
        };
        return off(parts) < off(than) && batches * (2 * parts + between) <= want + 1;
    };
    int by_groups = 0, by_heads = 1;
    while (half > 0 && by_groups < groups && nearer(by_groups + 1, by_groups)) ++by_groups;
    const bool cut = by_groups > 0;
    while (by_groups > 1 && static_cast<long long>(groups / by_groups) * G < 128) --by_groups;  // the least N of a job
    while (cut && nearer(2 * by_groups * by_heads, by_groups * by_heads) && 2 * by_heads <= half &&
           static_cast<long long>(half / (2 * by_heads)) * d * 2 >= kHostRowBytes)
        by_heads *= 2;
    for (int b = 0; b < batches; ++b) {
        HostChunk c;
        c.b0 = static_cast<int>(static_cast<long long>(B) * b / batches);
        c.bn = static_cast<int>(static_cast<long long>(B) * (b + 1) / batches) - c.b0;
        // heads whose groups stay together: all of them, or the KV head between the halves
        auto whole = [&](int kv0, int kvn) {
            c.kv0 = kv0, c.kvn = kvn, c.from[0] = 0, c.n[0] = N, c.from[1] = c.n[1] = 0, c.shift = G / 2;
            c.n_unshifted = H / 2 - kv0 * rep;
            return emit(c);
        };
        if (!cut) {
            if (const int rc = whole(0, Hkv)) return rc;
            continue;
        }
        for (int upper = 0; upper < 2; ++upper) {
            if (upper && Hkv > 2 * half)
                if (const int rc = whole(half, Hkv - 2 * half)) return rc;
            for (int h = 0; h < by_heads; ++h) {
                c.kv0 = (upper ? Hkv - half : 0) + half * h / by_heads;
                c.kvn = half * (h + 1) / by_heads - half * h / by_heads;
                for (int g = 0; g < by_groups; ++g) {
                    const int g0 = static_cast<int>(static_cast<long long>(groups) * g / by_groups);
                    const int g1 = static_cast<int>(static_cast<long long>(groups) * (g + 1) / by_groups);
                    c.from[0] = g0 * G, c.n[0] = (g1 - g0) * G, c.from[1] = c.n[1] = 0, c.shift = 0, c.n_unshifted = c.kvn * rep;
                    if (upper) {
                        c.from[0] += G / 2;
                        if (g1 == groups) {  // the group that wraps: the first G / 2 tokens and the last ones
                            c.shift = G / 2, c.n_unshifted = 0;
                            if (g0 == 0) c.from[0] = 0;
                            else c.from[1] = c.from[0], c.n[1] = c.n[0] - G / 2, c.from[0] = 0, c.n[0] = G / 2;
                        }
                    }
                    if (const int rc = emit(c)) return rc;
                }
            }
        }
    }
    return 0;
}

}  // namespace s2a
