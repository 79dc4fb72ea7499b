// Host check of the two integer forms of a single cell's Laplacian sum (lap6_units with lap6_rounded, and with its plain sum where
// that is exact) against the FP64 evaluation order: prints "cells accepted exact mismatches" over seeded random stencils.  The
// kernel picks a form per warp, so an exact cell also goes through lap6_rounded: every accepted cell is checked by both.
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
    long accepted = 0, exact = 0, mismatches = 0;
    for (long t = 0; t < n; ++t) {
        const int kind = (int)(next_u64() % 9);
        const double c = (next_u64() % 2 ? 1.0 : -1.0) * (1.0 + unif()) * ldexp(1.0, (int)(next_u64() % 2098) - 1075);
        double x[6], C = kind == 8 ? (next_u64() % 8 ? 0.0 : -0.0) : c;
        for (double& v : x) {
            const double r = 2.0 * unif() - 1.0;
            switch (kind) {
                case 0: v = c * (1.0 + 1e-3 * r); break;
                case 1: v = c * (1.0 + 1e-14 * r); break;
                case 2: v = c * (1.0 + 0.9 * r); break;                        // near a factor of two
                case 3: v = next_u64() % 3 ? c : c * (1.0 + 1e-6 * r); break;  // ties and zero differences
                case 4: v = c * (1.0 + 3.0 * r); break;                        // sign changes
                case 5: v = c * exp(3.0 * r); break;                           // exponents up to 4 apart: rounded partial sums
                case 6: v = hg::bits_d(hg::dbits(c) + (int64_t)(next_u64() % 64) - 32); break;
                case 7: v = ldexp(c, (int)(next_u64() % 9) - 4); break;        // the border of the accepted exponents
                default: {
                    const int w = (int)(next_u64() % 24);
                    v = w < 21 ? 0.0 : w == 21 ? -0.0 : w == 22 ? 0x1p-1074 * (double)(next_u64() % 5) : ldexp(r, -1070);
                }
            }
        }
        const hg::Lap6 k = hg::lap6_units(C, x[0], x[1], x[2], x[3], x[4], x[5]);
        if (!k.ok) continue;
        ++accepted;
        double L = (x[0] - C) + (x[1] - C);
        for (int i = 2; i < 6; ++i) L = L + (x[i] - C);
        mismatches += hg::dbits(hg::pack_units(hg::lap6_rounded(k.D), k.h)) != hg::dbits(L);
        if (!k.exact) continue;
        ++exact;
        mismatches += hg::dbits(hg::pack_units(k.S, k.h)) != hg::dbits(L);
    }
    printf("%ld %ld %ld %ld\n", n, accepted, exact, mismatches);
    return 0;
}
