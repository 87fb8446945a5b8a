// Host-side check of FastDiv and BlockOrder (s2a_params.h): divisors and dividends at the edges of their range
// against the division itself.  Prints "ok" and returns 0, or says what failed.
#include <cstdio>
#include <initializer_list>

#include "s2a_params.h"

using namespace s2a;

int main() {
    const int top = 0x7fffffff;
    unsigned long long x = 88172645463325252ull;  // xorshift
    auto next = [&] { return x ^= x << 13, x ^= x >> 7, x ^= x << 17, static_cast<int>(x & top); };
    auto check = [&](int n, int d) {
        int rest;
        return FastDiv(d)(n) == n / d && FastDiv(d)(n, &rest) == n / d && rest == n % d;
    };
    for (int i = 0; i < 300000; ++i) {
        const int shift = i % 31, some = next() >> shift, d = some > 0 ? some : 1;
        for (int n : {next(), 0, top, d - 1, d, top - top % d, top - top % d - 1})
            if (!check(n, d)) return std::printf("FAIL %d / %d\n", n, d), 1;
    }
    for (int units : {1, 5, 8, 9, 100})
        for (int tiles : {1, 3, 16})
            for (int chunk : {1, 2, 8, 64}) {
                const BlockOrder order(units, tiles, chunk);
                for (int idx = 0; idx < units * tiles; ++idx) {
                    const int c = chunk < units ? chunk : units, first = idx / (c * tiles) * c, within = idx % (c * tiles);
                    const int in = units - first < c ? units - first : c;
                    int unit, rank;
                    order.decode(idx, &unit, &rank);
                    if (unit != first + within % in || rank != within / in) return std::printf("FAIL order %d %d %d: %d\n", units, tiles, chunk, idx), 1;
                }
            }
    std::printf("ok\n");
    return 0;
}
