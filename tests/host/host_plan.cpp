// Host-side check of cut_host_job (host_plan.h): over edge shapes every (batch item, KV head, token) is in exactly
// one chunk, every chunk's groups are the whole job's groups, and a chunk is a job that the entry points take.
// Prints "ok" and returns 0, or says what failed.
#include <cstdio>
#include <set>
#include <vector>

#include "host_plan.h"

using namespace s2a;

int main() {
    const int heads[][2] = {{2, 1}, {4, 4}, {6, 3}, {8, 2}, {10, 5}, {32, 32}, {40, 40}, {64, 8}};
    int most = 0;
    for (const auto& hh : heads)
        for (int d : {64, 128})
            for (int B : {1, 2, 5, 40})
                for (int G : {8, 128, 200, 1000, 2048})
                    for (int groups : {1, 2, 3, 4, 17, 64}) {
                        const int H = hh[0], Hkv = hh[1], N = G * groups, rep = H / Hkv;
                        if (N < 128 || 1LL * B * N * Hkv > (4 << 20)) continue;
                        std::vector<char> seen(static_cast<size_t>(B) * Hkv * (N / 4));
                        int chunks = 0, wide = 0;
                        const int rc = cut_host_job(B, N, H, Hkv, d, G, [&](const HostChunk& c) {
                            const int n = c.tokens();
                            if (n < 128 || n % G != 0 || c.bn < 1 || c.kvn < 1 || (c.bn > 1 && c.n[0] != N)) return 1;
                            if (c.shift != 0 && c.shift != G / 2) return 2;
                            // token of every place of the chunk's rows
                            std::vector<int> tok(n);
                            for (int i = 0; i < n; ++i) tok[i] = i < c.n[0] ? c.from[0] + i : c.from[1] + i - c.n[0];
                            for (int b = c.b0; b < c.b0 + c.bn; ++b)
                                for (int kv = c.kv0; kv < c.kv0 + c.kvn; ++kv)
                                    for (int i = 0; i < n; i += 4) {
                                        if (tok[i] < 0 || tok[i] + 3 >= N || tok[i + 3] != tok[i] + 3) return 3;
                                        char& s = seen[(static_cast<size_t>(b) * Hkv + kv) * (N / 4) + tok[i] / 4];
                                        if (s) return 4;
                                        s = 1;
                                    }
                            for (int h = c.kv0 * rep; h < (c.kv0 + c.kvn) * rep; ++h) {
                                const int s_job = h < H / 2 ? 0 : G / 2, s_chunk = h - c.kv0 * rep < c.n_unshifted ? 0 : c.shift;
                                for (int p = 0; p < n; p += 4) {  // place p of the shifted order of the chunk
                                    const int at = (p + s_chunk) % n, first = (p / G * G + s_chunk) % n;
                                    const int in_group = (tok[at] - s_job + N) % N % G;
                                    if (in_group != p % G || (tok[at] - s_job + N) % N / G != (tok[first] - s_job + N) % N / G) return 5;
                                    // and the wrap is where the job's wrap is
                                    if (p % G != 0 && (at < (p - 4 + s_chunk) % n) != (tok[at] < tok[(p - 4 + s_chunk) % n])) return 6;
                                }
                            }
                            ++chunks, wide += c.n[0] == N;
                            return 0;
                        });
                        for (char s : seen)
                            if (rc || !s) return std::printf("FAIL rc %d B %d G %d groups %d H %d Hkv %d d %d\n", rc, B, G, groups, H, Hkv, d), 1;
                        if (chunks > kHostChunks + 1) return std::printf("FAIL %d chunks\n", chunks), 1;
                        if (chunks > most) most = chunks;
                    }
    // the number of chunks, for sizes that call for all of them too
    for (const auto& hh : heads)
        for (int d : {64, 128})
            for (int B = 1; B <= 33; ++B)
                for (int N : {1024, 8192, 32768, 131072})
                    for (int groups : {1, 4, 5, 16}) {
                        if (N % (8 * groups) != 0) continue;
                        int chunks = 0;
                        cut_host_job(B, N, hh[0], hh[1], d, N / groups, [&](const HostChunk&) { return ++chunks, 0; });
                        if (chunks > kHostChunks + 1)
                            return std::printf("FAIL %d chunks: B %d N %d groups %d H %d Hkv %d d %d\n", chunks, B, N, groups, hh[0], hh[1], d), 1;
                        if (chunks > most) most = chunks;
                    }
    if (most < kHostChunks) return std::printf("FAIL at most %d chunks\n", most), 1;
    std::printf("ok\n");
    return 0;
}
