// Host-side check of the integer hand-over between tensor-core passes (emu.cuh:
// requantize), compiled and run by tests/test_emu_requantize.py on the CPU: for
// integers below 2^60 of scales up to 100 binades below the line's, the result is the
// exactly rounded shift plus the digit bias, and its 10-bit fields are the digits that
// digits() gives.  Prints OK and returns 0 when every check passes.
#include <cstdio>
#include <random>

#include "emu.cuh"

using namespace wvl::emu;

int main() {
    std::mt19937_64 rng(9041543);
    int fails = 0;
    for (int it = 0; it < 2000000; ++it) {
        const int bits = 1 + (int)(rng() % 60);
        long long t = (long long)(rng() >> (64 - bits));
        if (it % 7 == 0) t = (1LL << bits) - 1 - (it % 14 == 0);
        if (it % 11 == 0 && bits > 1) t = 1LL << (bits - 1);
        if (rng() & 1) t = -t;
        const int g = (int)(rng() % 2000) - 1000;
        const int E = g + (int)(rng() % 101) + (bits > HAND_MIN ? bits : HAND_MIN);
        // round half up of t 2^(g + QBITS - E), in 128 bits
        const int sh = E - QBITS - g + 8;   // of 2^8 t, >= 1
        const __int128 half = (__int128)1 << (sh > 110 ? 0 : sh - 1);
        const __int128 X = sh > 110 ? 0 : (((__int128)t << 8) + half) >> sh;
        const long long Y = requantize(t, g, E);
        bool ok = (__int128)Y == X + DBIAS && Y >= 0;
        int d[S];
        digits((long long)X, d);
        for (int q = 1; q < S; ++q) ok = ok && (int)((Y >> (DBITS * (S - 1 - q))) & 1023) - 512 == d[q];
        ok = ok && (int)(Y >> (DBITS * (S - 1))) - 512 == d[0] && d[0] >= -512 && d[0] <= 512;
        if (!ok && fails++ < 10) std::printf("FAIL t %lld g %d E %d\n", t, g, E);
    }
    if (fails == 0) std::printf("OK\n");
    return fails != 0;
}
