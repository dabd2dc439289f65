// Host-side check of the hand-over between tensor-core passes on a line's own scale
// (emu.cuh), compiled and run by tests/test_emu_handover.py on the CPU:
//  - requantize() where the line's largest value lies below the scale of an integer, so that
//    the shift goes to the left, is exact: X = t 2^(g + QBITS - E);
//  - hand_bits() bounds an integer's magnitude, by less than a factor of four;
//  - every line of n elements is covered by hand_slots(n) warps of 32 source lines at most,
//    each writing one slot of its own, and the slots, scales and line exponents of an
//    operator's passes fit into one FP64 array of the cell, for any extents.
// Prints OK and returns 0 when every check passes.
#include <cstdio>
#include <random>
#include <set>

#include "emu.cuh"

using namespace wvl::emu;

int main() {
    std::mt19937_64 rng(20090415);
    int fails = 0;
    for (int it = 0; it < 2000000; ++it) {
        const int bits = 1 + (int)(rng() % HAND_MIN);
        long long t = (long long)(rng() >> (64 - bits));
        if (it % 5 == 0) t = 1LL << bits;   // the bound itself
        if (rng() & 1) t = -t;
        const int g = (int)(rng() % 2000) - 1000;
        const int E = g + bits;   // |t| 2^g <= 2^E, E - g <= HAND_MIN
        const __int128 X = (__int128)t << (g + QBITS - E);
        const long long Y = requantize(t, g, E);
        bool ok = (__int128)Y == X + DBIAS && Y >= 0;
        int d[S];
        digits((long long)X, d);
        for (int q = 1; q < S; ++q) ok = ok && (int)((Y >> (DBITS * (S - 1 - q))) & 1023) - 512 == d[q];
        ok = ok && (int)(Y >> (DBITS * (S - 1))) - 512 == d[0] && d[0] >= -512 && d[0] <= 512;
        if (!ok && fails++ < 10) std::printf("FAIL t %lld g %d E %d\n", t, g, E);
    }
    for (int E = -960; E < 1000; E += 7)   // zeros of lines of any other scale
        for (int g = -1100; g < 1000; g += 13)
            if (requantize(0, g, E) != DBIAS && fails++ < 10) std::printf("FAIL zero g %d E %d\n", g, E);
    for (int it = 0; it < 2000000; ++it) {   // the exponent of an integer, a tight upper bound
        const int bits = 1 + (int)(rng() % 60);
        long long t = (long long)(rng() >> (64 - bits));
        if (it % 3 == 0) t = (1LL << bits) - (it % 2);
        if (t == 0) continue;
        const int b = hand_bits((float)(rng() & 1 ? -t : t));
        if ((__int128)t > (__int128)1 << b || (__int128)4 * t <= (__int128)1 << b)
            if (fails++ < 10) std::printf("FAIL bits t %lld b %d\n", t, b);
    }
    if (hand_bits(0.f) != -126) ++fails;
    for (int n = 2; n <= 1024; n += 2) {
        // lines c of n source lines each: the warps that share one, and their slots
        for (int c = 0; c < 40; ++c) {
            std::set<int> used;
            for (int a = c * n; a < (c + 1) * n; ++a) used.insert(a / 32 - c * n / 32);
            if (*used.begin() != 0 || *used.rbegin() >= hand_slots(n) || (int)used.size() != *used.rbegin() + 1)
                if (fails++ < 10) std::printf("FAIL slots n %d c %d\n", n, c);
        }
        // four arrays (exponents of passes 2 and 3, scales of pass 1, line exponents or scales
        // of pass 2), each of at most half the cell's points in ints
        if (2 * hand_slots(n) > n && fails++ < 10) std::printf("FAIL size n %d\n", n);
    }
    if (fails == 0) std::printf("OK\n");
    return fails != 0;
}
