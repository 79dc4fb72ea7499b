// Host check of lap6_units2 (two cells along x in common units) against the FP64 evaluation order: prints
// "cells accepted mismatches" over seeded random stencils of several kinds.
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>

#include "../../paper_1602_05700_gb300/csrc/lap_int.cuh"

static uint64_t state;
static uint64_t next_u64() {  // splitmix64
    uint64_t z = (state += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
static double unif() { return (double)(next_u64() >> 11) * 0x1.0p-53; }

int main(int argc, char** argv) {
    const long n = argc > 1 ? atol(argv[1]) : 1000000;
    state = argc > 2 ? strtoull(argv[2], 0, 10) : 1;
    long cells = 0, accepted = 0, mismatches = 0;
    for (long t = 0; t < n; ++t) {
        const int kind = (int)(next_u64() % 8);
        const double base = (next_u64() % 2 ? 1.0 : -1.0) * (1.0 + unif()) * ldexp(1.0, (int)(next_u64() % 2098) - 1075);
        auto value = [&]() -> double {
            const double r = 2.0 * unif() - 1.0;
            switch (kind) {
                case 0: return base * (1.0 + 1e-3 * r);
                case 1: return base * (1.0 + 1e-14 * r);
                case 2: return base * (1.0 + 0.9 * r);
                case 3: return next_u64() % 3 ? base : base * (1.0 + 1e-6 * r);
                case 4: return base * (1.0 + 3.0 * r);
                case 5: return base * exp(2.0 * r);
                case 6: return hg::bits_d(hg::dbits(base) + (int64_t)(next_u64() % 64) - 32);
                default: {
                    const int w = (int)(next_u64() % 24);
                    return w < 20 ? 0.0 : w == 20 ? -0.0 : w == 21 ? 0x1p-1074 * (double)(next_u64() % 5) : ldexp(r, -1070);
                }
            }
        };
        double c[2] = {value(), value()}, v[2][6];
        for (int q = 0; q < 2; ++q)
            for (int i = 0; i < 6; ++i) v[q][i] = value();
        v[0][1] = c[1];
        v[1][0] = c[0];
        const hg::Lap6Pair k = hg::lap6_units2(c, v);
        for (int q = 0; q < 2; ++q) {
            ++cells;
            if (!k.ok) continue;
            ++accepted;
            double L = (v[q][0] - c[q]) + (v[q][1] - c[q]);
            for (int i = 2; i < 6; ++i) L = L + (v[q][i] - c[q]);
            const double r = hg::pack_units(hg::lap6_rounded(k.D[q]), k.h);
            mismatches += hg::dbits(r) != hg::dbits(L);
            if (k.exact) mismatches += hg::dbits(hg::pack_units(k.S[q], k.h)) != hg::dbits(L);
        }
    }
    printf("%ld %ld %ld\n", cells, accepted, mismatches);
    return 0;
}
