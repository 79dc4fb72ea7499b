// The FP64 Laplacian sum of the sub-step, L = (((((xl-c) + (xr-c)) + (ys-c)) + (yn-c)) + (zm-c)) + (zp-c) with
// every difference and every partial sum rounded to double (the plain evaluation order of Eq. HNeq's discretisation,
// Sec. 2), computed with integer instructions that give the same bits.
//
// Why: GB300 executes FP64 arithmetic at about 2 operations per SM and clock (16 cycles per warp instruction), while
// its integer pipes take 64 lanes per clock; the 11 FP64 operations of L are most of an FP64 sub-step's 15.
//
// Units: let e be the smallest biased exponent of the seven values and u = 2^(e - 1075) its unit in the last place.  If all
// seven have one sign, 64 <= e <= 1993 and no exponent exceeds e + 7, each value is an integer below 2^60 times u, so
// every difference and every sum of differences is an exact integer below 2^63, and u >= 2^-1011 keeps every
// rounded result normal.  An operation of the FP64 order is then the rounding of an exact integer to 53 significant
// bits, to nearest even:
//   * an integer of magnitude at most 2^53 is unchanged.  Where that holds for all six differences and all five partial
//     sums (any field whose neighbours lie within a factor of about two: potentials, and the steep tails of compact
//     sources too), L is the plain integer sum;
//   * otherwise each operation is rounded as it is made (round53).
// A zero result is +0, as x - x and a + (-a) are in round-to-nearest.  A cell and six neighbours that are all +0 give
// L = +0 as well.  Other stencils (sign changes, exponents further apart, subnormals) are left to FP64.
#pragma once

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif
#ifndef __CUDA_ARCH__
#include <string.h>
#endif

namespace hg {

constexpr unsigned long long kFrac52 = (1ull << 52) - 1;
constexpr unsigned long long kHidden52 = 1ull << 52;

__host__ __device__ __forceinline__ unsigned long long dbits(double x) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(x);
#else
    unsigned long long u;
    memcpy(&u, &x, sizeof u);
    return u;
#endif
}

__host__ __device__ __forceinline__ double bits_d(unsigned long long u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double x;
    memcpy(&x, &u, sizeof x);
    return x;
#endif
}

__host__ __device__ __forceinline__ int clz64(unsigned long long v) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}

__host__ __device__ __forceinline__ unsigned umin3(unsigned a, unsigned b, unsigned c) {
#ifdef __CUDA_ARCH__
    return __vimin3_u32(a, b, c);
#else
    const unsigned m = a < b ? a : b;
    return m < c ? m : c;
#endif
}
__host__ __device__ __forceinline__ unsigned umax3(unsigned a, unsigned b, unsigned c) {
#ifdef __CUDA_ARCH__
    return __vimax3_u32(a, b, c);
#else
    const unsigned m = a > b ? a : b;
    return m > c ? m : c;
#endif
}

// the significand of a double, hidden bit set, shifted left by d & 7 (on the device d is taken modulo 32 by the funnel
// shift: only d <= 7 is used)
__host__ __device__ __forceinline__ long long significand(unsigned long long b, unsigned d) {
#ifdef __CUDA_ARCH__
    const unsigned lo = (unsigned)b, hi = ((unsigned)(b >> 32) & 0xfffffu) | 0x100000u;
    return (long long)(((unsigned long long)__funnelshift_l(lo, hi, d) << 32) | __funnelshift_l(0u, lo, d));
#else
    return (long long)(((b & kFrac52) | kHidden52) << (d & 7u));
#endif
}

// the six differences in units of the stencil's smallest ulp, and which of the forms above serve it
struct Lap6 {
    long long D[6];
    long long S;   // their plain sum: L in units u when `exact`
    unsigned h;    // sign and smallest biased exponent
    bool exact;    // no operation of the FP64 order rounds
    bool ok;       // the integer forms hold
};

// hi word of |v|, up to one: v ^ (v >> 63), so a magnitude of at most 2^53 leaves the bits from 2^21 on clear
__host__ __device__ __forceinline__ unsigned mag_hi(long long v) {
    const int h = (int)(v >> 32);
    return (unsigned)(h ^ (h >> 31));
}

__host__ __device__ __forceinline__ Lap6 lap6_units(double c, double x0, double x1, double x2, double x3, double x4,
                                                    double x5) {
    const unsigned long long b[7] = {dbits(x0), dbits(x1), dbits(x2), dbits(x3), dbits(x4), dbits(x5), dbits(c)};
    unsigned h[7];
#pragma unroll
    for (int i = 0; i < 7; ++i) h[i] = (unsigned)(b[i] >> 52);
    const unsigned lo = umin3(umin3(h[0], h[1], h[2]), umin3(h[3], h[4], h[5]), h[6]);
    const unsigned hi = umax3(umax3(h[0], h[1], h[2]), umax3(h[3], h[4], h[5]), h[6]);
    Lap6 r;
    r.h = lo;
    const bool near = hi - lo <= 7u;  // exponents within 7, and one sign (else hi - lo >= 2^11 - 2046)
    const long long C = significand(b[6], h[6] - lo);
    unsigned acc = 0;
    r.S = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        r.D[i] = significand(b[i], h[i] - lo) - C;
        r.S += r.D[i];
        acc |= mag_hi(r.D[i]) | mag_hi(r.S);
    }
    // all +0: the hidden bits cancel, every difference is 0 (a positive subnormal's is positive, so S = 0 tells)
    r.ok = near && (((lo & 0x7ffu) - 64u <= 1993u - 64u) || (b[6] == 0ull && r.S == 0));
    r.exact = r.ok && acc < (1u << 21);
    return r;
}

// The values at p and p + 1 (p on 16 bytes), or the one at p twice where `two` is false: behind the last cell of an odd row lies
// the +x ghost, which another thread of the launch may be writing, so it is not read there.
__host__ __device__ __forceinline__ void load_pair(const double* p, bool two, double (&v)[2]) {
    if (two) {
#ifdef __CUDA_ARCH__
        const double2 x = *reinterpret_cast<const double2*>(p);
        v[0] = x.x;
        v[1] = x.y;
#else
        v[0] = p[0];
        v[1] = p[1];
#endif
    } else {
        v[0] = v[1] = p[0];
    }
}

// Two cells next to each other along x in common units (the smallest ulp of their twelve values): the conversions of c0, c1
// and their difference serve both.  v[q]: the neighbours of cell q in the order of the sum (v[0][1] is c1, v[1][0] is c0).
struct Lap6Pair {
    long long D[2][6];
    long long S[2];
    unsigned h;
    bool exact, ok;
};
__host__ __device__ __forceinline__ Lap6Pair lap6_units2(const double (&c)[2], const double (&v)[2][6]) {
    const unsigned long long b[12] = {dbits(c[0]),    dbits(c[1]),    dbits(v[0][0]), dbits(v[1][1]),
                                      dbits(v[0][2]), dbits(v[0][3]), dbits(v[0][4]), dbits(v[0][5]),
                                      dbits(v[1][2]), dbits(v[1][3]), dbits(v[1][4]), dbits(v[1][5])};
    unsigned h[12];
#pragma unroll
    for (int i = 0; i < 12; ++i) h[i] = (unsigned)(b[i] >> 52);
    const unsigned lo = umin3(umin3(umin3(h[0], h[1], h[2]), umin3(h[3], h[4], h[5]), umin3(h[6], h[7], h[8])),
                              umin3(h[9], h[10], h[11]), h[0]);
    const unsigned hi = umax3(umax3(umax3(h[0], h[1], h[2]), umax3(h[3], h[4], h[5]), umax3(h[6], h[7], h[8])),
                              umax3(h[9], h[10], h[11]), h[0]);
    Lap6Pair r;
    r.h = lo;
    const bool near = hi - lo <= 7u;
    long long m[12];
#pragma unroll
    for (int i = 0; i < 12; ++i) m[i] = significand(b[i], h[i] - lo);
    const long long D01 = m[1] - m[0];
    r.D[0][0] = m[2] - m[0];
    r.D[0][1] = D01;
    r.D[1][0] = -D01;
    r.D[1][1] = m[3] - m[1];
    unsigned acc = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
#pragma unroll
        for (int i = 0; i < 4; ++i) r.D[q][2 + i] = m[4 + 4 * q + i] - m[q];
        r.S[q] = 0;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            r.S[q] += r.D[q][i];
            acc |= mag_hi(r.D[q][i]) | mag_hi(r.S[q]);
        }
    }
    // all +0 as in lap6_units: with c0 = c1 = +0 no difference is negative
    r.ok = near && (((lo & 0x7ffu) - 64u <= 1993u - 64u) || ((b[0] | b[1]) == 0ull && r.S[0] == 0 && r.S[1] == 0));
    r.exact = r.ok && acc < (1u << 21);
    return r;
}

// an integer rounded to 53 significant bits, to nearest even
__host__ __device__ __forceinline__ long long round53(long long v) {
    if (mag_hi(v) < (1u << 21)) return v;
    const unsigned long long A = (unsigned long long)(v < 0 ? -v : v);
    const int k = 11 - clz64(A);  // bits beyond 53 (A = 2^53 itself has one, and drops a zero)
    const unsigned long long rem = A & ((1ull << k) - 1), half = 1ull << (k - 1);
    unsigned long long q = A >> k;
    q += (rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull;
    const long long m = (long long)(q << k);
    return v < 0 ? -m : m;
}

// L in units u with every operation rounded as the FP64 order rounds it (valid when ok)
__host__ __device__ __forceinline__ long long lap6_rounded(const long long (&D)[6]) {
    long long P = round53(round53(D[0]) + round53(D[1]));
#pragma unroll
    for (int i = 2; i < 6; ++i) P = round53(P + round53(D[i]));
    return P;
}

// S u with u = 2^(e - 1075), h the sign and biased exponent e; S has at most 53 significant bits and |S| < 2^63: with lz
// leading zeros |S| 2^lz has its top bit at 63, so |S| = mant 2^(11 - lz) with mant = (|S| 2^lz) 2^-11 in [2^52, 2^53), and the
// biased exponent is e + 11 - lz (mant's hidden bit adds the last 1); the sign is h's times S's; 0 gives +0
__host__ __device__ __forceinline__ double pack_units(long long S, unsigned h) {
    const unsigned long long A = (unsigned long long)(S < 0 ? -S : S);
    const int lz = clz64(A);
    const unsigned long long mant = (A << (lz & 63)) >> 11;
    const unsigned sign = ((h << 20) ^ (unsigned)((unsigned long long)S >> 32)) & 0x80000000u;
    const unsigned long long top = (unsigned long long)(sign | (((h & 0x7ffu) + 10u - (unsigned)lz) << 20)) << 32;
    return A == 0 ? 0.0 : bits_d(top + mant);
}

// The next two are entry points of the host checks only (the sub-steps vote on a form per warp, cell.cuh).
// L from integers; false when the stencil is left to FP64 (then L is not set)
__host__ __device__ __forceinline__ bool lap6_int(double c, double x0, double x1, double x2, double x3, double x4,
                                                  double x5, double& L) {
    const Lap6 k = lap6_units(c, x0, x1, x2, x3, x4, x5);
    if (k.ok) L = pack_units(k.exact ? k.S : lap6_rounded(k.D), k.h);
    return k.ok;
}

// the six differences from integers; false (d not set) when the stencil is left to FP64
__host__ __device__ __forceinline__ bool lap6_diffs(double c, double x0, double x1, double x2, double x3, double x4,
                                                    double x5, double (&d)[6]) {
    const Lap6 k = lap6_units(c, x0, x1, x2, x3, x4, x5);
    if (k.ok) {
#pragma unroll
        for (int i = 0; i < 6; ++i) d[i] = pack_units(round53(k.D[i]), k.h);
    }
    return k.ok;
}

// t = 2c - prev rounded once to nearest-even (the leapfrog's first operation), from integers where c is normal in the
// range above and prev has c's sign, an exponent within one of c's and |prev| < 2|c|: in units u = 2^(e_c - 1076),
// T = 4 M_c - M_prev 2^(e_prev - e_c + 1) is a positive integer below 2^55, rounded here to 53 significant bits.
// c = prev = +0 gives +0.  Otherwise false (t not set).
__host__ __device__ __forceinline__ bool twice_minus_int(double c, double prev, double& t) {
    const unsigned long long cb = dbits(c), pb = dbits(prev);
    const unsigned hc = (unsigned)(cb >> 52);
    const unsigned ec = hc & 0x7ffu;
    const unsigned d = (unsigned)(pb >> 52) - hc + 1u;
    const long long T = (long long)(((cb & kFrac52) | kHidden52) << 2) -
                        (long long)(((pb & kFrac52) | kHidden52) << (d & 3u));
    const unsigned long long Tu = (unsigned long long)T;
    const int k = 11 - clz64(Tu);  // significant bits beyond 53 (negative: room to shift left)
    unsigned long long q;
    if (k > 0) {
        const unsigned long long rem = Tu & ((1ull << k) - 1), half = 1ull << (k - 1);
        q = Tu >> k;
        q += (rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull;  // q = 2^53 carries into the exponent
    } else {
        q = Tu << ((-k) & 63);
    }
    const unsigned long long e = (unsigned long long)((int)ec + k - 1);  // biased exponent of the result
    t = (cb | pb) == 0ull ? 0.0 : bits_d((cb & (1ull << 63)) | (((e - 1ull) << 52) + q));
    return (cb | pb) == 0ull || (d <= 2u && T > 0 && ec >= 64u && ec <= 2000u);
}

}  // namespace hg
