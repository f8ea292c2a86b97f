// Host check of lbmfx::from_fixed_int (lbm_f64fx.cuh): the conversion on the integer pipes gives
// the bits of from_fixed (one round-to-nearest-even conversion, then the exponent moves) for every
// 64-bit value below 2^63 in magnitude: all powers of two and their neighbours, ties and their
// neighbours at every bit length, random values of every length.
//
// usage: fxconv_check <cases> <seed>; the last line reads "<n> cases, <m> failures".
#include <cstdio>
#include <cstdlib>

#include "../../paper_2408_01081_gb300/csrc/lbm_f64fx.cuh"

using lbmfx::i64;
using lbmfx::u64;

static long cases = 0, fails = 0;

static void check(u64 mag, int E)
{
    if (mag >> 63) return;
    const int add = (E - 1081) * (1 << 20);
    for (int s = 0; s < 2; ++s) {
        const i64 y = s ? -(i64)mag : (i64)mag;
        ++cases;
        if (lbmfx::from_fixed(y, add) != lbmfx::from_fixed_int(y, add) && ++fails < 10)
            std::printf("%lld E %d: %016llx %016llx\n", y, E, lbmfx::from_fixed(y, add), lbmfx::from_fixed_int(y, add));
    }
}

int main(int argc, char** argv)
{
    const long n = argc > 1 ? std::atol(argv[1]) : 100000;
    u64 st = argc > 2 ? std::strtoull(argv[2], nullptr, 10) : 1;
    const int Es[3] = {59, 1023, 2042};
    for (int e = 0; e < 3; ++e) {
        for (int b = 0; b < 63; ++b)
            for (int d = -3; d <= 3; ++d) check((1ull << b) + (u64)(i64)d, Es[e]);
        for (int b = 53; b < 63; ++b)                  // ties: an odd multiple of half the last kept bit
            for (u64 q = (1ull << 52); q < (1ull << 52) + 4; ++q)
                for (int d = -1; d <= 1; ++d) {
                    const int drop = b - 52;
                    check((q << drop) + (1ull << (drop - 1)) + (u64)(i64)d, Es[e]);
                    check(((q | 0xFFFFFFFFFFFF0ull) << drop) + (1ull << (drop - 1)) + (u64)(i64)d, Es[e]);
                }
    }
    for (long c = 0; c < n; ++c) {
        u64 z = (st += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z ^= z >> 27;
        check(z >> (1 + (c % 63)), Es[c % 3]);
    }
    std::printf("%ld cases, %ld failures\n", cases, fails);
    return fails != 0;
}
