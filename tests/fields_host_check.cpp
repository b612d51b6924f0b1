// The integer conversion of a 2^-58 fixed-point number to the nearest double (lbm_df.cuh),
// built for the host, against the hardware's conversion of the 64-bit integer.
#include <cstdio>
#include <cstdint>
#include <cmath>
#include <random>

#include "../paper_1611_02445_gb300/csrc/lbm_df.cuh"

int main() {
    std::mt19937_64 rng(5);
    long bad = 0;
    auto check = [&](int64_t x) {
        const double ref = std::ldexp((double)x, -58);
        if (lbm::bits_of(lbm::fix_to_double(x)) != lbm::bits_of(ref)) bad++;
    };
    for (int64_t s : {0ll, 1ll, -1ll, 2ll, 3ll}) check(s);
    // every length, with the roundings that tie, round up into the next binade and down
    for (int len = 1; len < 63; len++) {
        const int64_t top = 1ll << len;
        for (int64_t d = -3; d <= 3; d++) {
            check(top + d);
            check(-(top + d));
        }
        if (len > 53) {
            const int64_t half = 1ll << (len - 53), ulp = half << 1;
            for (int64_t k = 0; k < 4; k++)
                for (int64_t e = -1; e <= 1; e++) {
                    check(top + k * ulp + half / 2 + e);
                    check(top + k * half + e);
                    check(2 * top - 1 - k * (half / 2) - e > 0 ? 2 * top - 1 - k * (half / 2) - e : top);
                }
        }
    }
    for (int i = 0; i < 1000000; i++) {
        const int64_t x = (int64_t)(rng() >> (1 + i % 62));
        check(i & 1 ? -x : x);
    }
    std::printf("%ld\n", bad);
    return 0;
}
