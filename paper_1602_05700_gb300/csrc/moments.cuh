// FP64 multipole moments of a density, Q_lm = sum_cells rho h^3 r^l Y_lm(x) (arXiv 1602.05700, Sec. 4: Dirichlet boundary by
// multipole expansion), by way of the Cartesian moments M_abc = sum rho X^a Y^b Z^c, a + b + c <= lmax.
//
// What bounds it: the FP64 pipe (2 lanes per SM and clock).  Evaluating the harmonics of every cell and adding each to
// a double-double sum costs about 240 FP64 operations per cell at lmax = 4 (9.3 ms at 256^3, against 1.5 ms for the 20
// sub-steps that follow).  r^l Y_lm is a homogeneous polynomial with integer coefficients up to one factor, so the sums can
// be taken axis by axis and the harmonics formed once per block:
//   * a lane owns a row (fixed j, k), or a part of one, and sums rho X^a over it, four cells at a time in plain FP64 and from
//     there on in double-double (T_a; the rounding error of one addition starts the next four cells' sum): 9 operations
//     per cell at lmax = 4.  X is the same for all lanes, so its powers come from a table in shared memory, each rounded
//     once;
//   * T_a times Z^c goes to the lane's sums over k (10 per row and (a, c)); Y^b, a transposing warp reduction (31 merges
//     per 32 moments), the sum over warps and the change to Q_lm follow once per block.  Y^b and Z^c are pairs.
// Coordinates are half cells counted from the integer one nearest the expansion origin, so a term is no larger than the moment
// it belongs to (counted from the grid's centre, a compact source at an origin off the centre lost (distance / radius)^l of its
// accuracy: 7e6 units of 2^-53 sum |rho| |x|^l at l = 8), the powers are integers (exact up to 2^53) and the cancellation inside
// a harmonic (x^2 - y^2 of a round source) holds.  The Cartesian moments stay pairs through the shift by the remaining half
// cell or less to the origin and the change to Q_lm.
// Lanes read rows of their own, 16 cells at a time and a group ahead: the sectors are used whole out of L1.  Float input
// becomes double by integer instructions (exact), since conversions are slow as well; groups of zeros (vacuum around the
// source) are skipped.
//
// Measured (random density, a call of hg_moments_noalloc with both its launches, us, harmonics per cell -> this): lmax 4:
// 32^3 347 -> 73, 128^3 1475 -> 114, 256^3 9490 -> 413, 512^3 73,500 -> 2500; lmax 8: 256^3 30,030 -> 852; lmax 0: 256^3 374 ->
// 116.  (With the errors summed beside T_a: 449 at 256^3 and lmax 4; sums of 16 cells in plain FP64 about the grid's
// centre: 407, 512^3 2083.)  Error in units of 2^-53 sum |rho| |x|^l over spheres, Gaussians, constants and noise, centred or up
// to 0.8 of the way to a face, lmax 4 and 8 (the kernel's order evaluated on the host against quad precision; harmonics per
// cell with an exact sum -> this): largest 0.74 -> 0.44.
#pragma once

#include "cell.cuh"
#include "hg_internal.cuh"

namespace hg {

constexpr int kMomBlocks = 152;  // fixed, so that the result does not depend on the device
constexpr int kMomWarps = 8;

// number of monomials x^a y^b z^c with a + b + c < l, i.e. the index of the first one of degree l
__host__ __device__ constexpr int mono_off(int l) { return l * (l + 1) * (l + 2) / 6; }
// index of x^(l-b-c) y^b z^c among those of degree l
__host__ __device__ constexpr int mono_at(int l, int b, int c) { return c * (l + 1) - c * (c - 1) / 2 + b; }
constexpr int kMonoMax = (kMaxL + 1) * (kMaxL + 2) / 2;  // monomials of degree kMaxL

// 2^l r^l Y_lm / n_lm as integer coefficients of the monomials of degree l:
//   q_l^m = (-1)^m 2^-l sum_k (-1)^k (2l-2k)! / (k! (l-k)! (l-2k-m)!) z^(l-2k-m) (x^2 + y^2 + z^2)^k
// (the expansion of the Legendre polynomial's m-th derivative) times C_m or S_m, C_m + i S_m = (x + i y)^m.
struct HarmonicTable {
    double c[kMaxQ][kMonoMax];
};
constexpr double cfact(int n) { return n < 2 ? 1.0 : n * cfact(n - 1); }
constexpr double cbinom(int n, int k) { return cfact(n) / (cfact(k) * cfact(n - k)); }
constexpr HarmonicTable make_harmonics() {
    HarmonicTable T{};
    for (int l = 0; l <= kMaxL; ++l)
        for (int m = -l; m <= l; ++m) {
            const int am = m < 0 ? -m : m;
            for (int k = 0; 2 * k + am <= l; ++k) {
                const double q = ((k + am) % 2 ? -1.0 : 1.0) * cfact(2 * l - 2 * k) /
                                 (cfact(k) * cfact(l - k) * cfact(l - 2 * k - am));
                for (int u = 0; u <= k; ++u)          // (x^2)^(k-u-v) (y^2)^u (z^2)^v
                    for (int v = 0; u + v <= k; ++v)
                        for (int p = m < 0 ? 1 : 0; p <= am; p += 2) {  // x^(am-p) y^p with i^p
                            const double s = (p / 2) % 2 ? -1.0 : 1.0;
                            T.c[l * l + l + m][mono_at(l, 2 * u + p, l - 2 * k - am + 2 * v)] +=
                                q * s * cbinom(am, p) * cbinom(k, u) * cbinom(k - u, v);
                        }
            }
        }
    return T;
}
static __device__ const HarmonicTable kHarmonics = make_harmonics();

// ---- double-double sums --------------------------------------------------------------------------------------
// Each moment is a sum over every cell (1.7e7 terms at 256^3).  A plain running or tree sum in FP64 carries a
// rounding error that the lossless scheme then carries, through the Dirichlet data, into phi; so every partial sum
// beyond four cells is kept as an unevaluated pair s + e (TwoSum: s is the rounded sum, e collects the exact rounding
// errors), whose error is of order n eps^2 of the sum of |terms|.
// s <- s + x, and its rounding error: TwoSum as FastTwoSum on the operands ordered by the high words of their magnitudes (so the
// first one's exponent is not the smaller): three FP64 operations and integer selects, where TwoSum takes six on the pipe that
// bounds the kernel.
__device__ __forceinline__ double sum_error(double& s, double x) {
    const bool swap = (__double2hiint(s) & 0x7fffffff) < (__double2hiint(x) & 0x7fffffff);
    const double a = swap ? x : s, b = swap ? s : x;
    s = __dadd_rn(a, b);
    return __dsub_rn(b, __dsub_rn(s, a));
}
__device__ __forceinline__ void dd_add(double& s, double& e, double x) { e = __dadd_rn(e, sum_error(s, x)); }
// (s, e) += (s2, e2), renormalised so that s is the rounded value of the pair
__device__ __forceinline__ void dd_merge(double& s, double& e, double s2, double e2) {
    dd_add(s, e, s2);
    e = __dadd_rn(e, e2);
    const double t = __dadd_rn(s, e);
    e = __dsub_rn(e, __dsub_rn(t, s));
    s = t;
}
// (s, e) += (a, ae) * (x, xe)
__device__ __forceinline__ void dd_fma(double& s, double& e, double a, double ae, double x, double xe = 0.0) {
    const double p = __dmul_rn(a, x);
    const double pe = __fma_rn(a, xe, __fma_rn(ae, x, __fma_rn(a, x, -p)));
    dd_add(s, e, p);
    e = __dadd_rn(e, pe);
}
__device__ __forceinline__ void dd_warp(double& s, double& e) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double s2 = __shfl_xor_sync(0xffffffffu, s, o), e2 = __shfl_xor_sync(0xffffffffu, e, o);
        dd_merge(s, e, s2, e2);
    }
}

__device__ __forceinline__ bool nonzero(float x) { return (__float_as_uint(x) << 1) != 0u; }
__device__ __forceinline__ bool nonzero(double x) { return (__double_as_longlong(x) << 1) != 0; }

constexpr int kMomGroup = 16;  // cells of a row loaded together
constexpr int kMomSum = 4;     // cells summed in plain FP64
constexpr int kMomStretch = 2048;  // most cells of a row in the table of powers (8 x 16 KB at lmax = 8)

// the 16 cells of a row from cell `start` on; those beyond `hi` are 0.  vec: the row starts on a 16-byte boundary and has a
// whole number of 16-byte words, so that a group inside it can be read in such words
__device__ __forceinline__ void mom_load(const float* __restrict__ row, int start, int hi, bool vec, float (&v)[kMomGroup]) {
    if (vec && start + kMomGroup <= hi) {
#pragma unroll
        for (int g = 0; g < kMomGroup; g += 4) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(row + start + g));
            v[g] = x.x, v[g + 1] = x.y, v[g + 2] = x.z, v[g + 3] = x.w;
        }
    } else {
#pragma unroll
        for (int e = 0; e < kMomGroup; ++e) v[e] = start + e < hi ? __ldg(row + start + e) : 0.f;
    }
}
__device__ __forceinline__ void mom_load(const double* __restrict__ row, int start, int hi, bool vec, double (&v)[kMomGroup]) {
    if (vec && start + kMomGroup <= hi) {
#pragma unroll
        for (int g = 0; g < kMomGroup; g += 2) {
            const double2 x = __ldg(reinterpret_cast<const double2*>(row + start + g));
            v[g] = x.x, v[g + 1] = x.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < kMomGroup; ++e) v[e] = start + e < hi ? __ldg(row + start + e) : 0.0;
    }
}

struct MomArgs {
    int nx, ny, nz;
    int seg;                   // cells of a row in one task (a multiple of 16)
    double h3[2];              // cell volume, as a pair
    double org[3];             // the integer half cell nearest the origin, counted from the grid's corner, per axis
    double off[3][2];          // offset of that half cell from the origin in half cells (at most 1/2), as a pair
    double hl[kMaxL + 1][2];   // (h / 4)^l as a pair: half cells and the table's 2^-l
    int centred;               // off is zero
};

// (p, pe) <- (p, pe) * X for an integer X: exact while the power is below 2^106
__device__ __forceinline__ void dd_power(double& p, double& pe, double X) {
    const double q = __dmul_rn(p, X);
    pe = __fma_rn(pe, X, __fma_rn(p, X, -q));
    p = q;
}

// per-block partial moments: partial[2 (block nq + q) + {0, 1}]
template <typename T, int LMAX>
__global__ void __launch_bounds__(32 * kMomWarps, 1) k_moments(const T* __restrict__ rho, bool vec, MomArgs P,
                                                               YlmNorm N, double* __restrict__ partial, int ch) {
    extern __shared__ __align__(16) double pw[];  // [a][ch], a < LMAX: X^(a+1) of the cells of a stretch of the rows
    constexpr int NQ = (LMAX + 1) * (LMAX + 1), NM = mono_off(LMAX + 1), NB = (NM + 31) / 32;
    __shared__ double wm[kMomWarps][NB * 32][2], tot[NM][2], moved[NM][2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int m = lane; m < NB * 32; m += 32) wm[warp][m][0] = wm[warp][m][1] = 0.0;
    // tasks: (segment of the rows, 32 rows, 1 plane), plane fastest; a warp takes a contiguous range, so that its rows stay the
    // same.  Boxes of fewer than 32 rows put as many planes side by side in a task (nk) as the lanes hold.  Rows are cut into
    // segments where there are fewer tasks than warps (mom_segment).
    const int nk = P.ny < 32 ? 32 / P.ny : 1, dk = P.ny < 32 ? lane / P.ny : 0, dj = lane - dk * P.ny;  // lane -> plane, row
    const int kt = (P.nz + nk - 1) / nk, jt = (P.ny + 31) / 32;
    const long long W = (long long)kMomBlocks * kMomWarps, w = (long long)blockIdx.x * kMomWarps + warp;
    for (int x0 = 0; x0 < P.nx; x0 += ch) {
        const int x1 = P.nx < x0 + ch ? P.nx : x0 + ch;
        if constexpr (LMAX > 0) {
            __syncthreads();  // the stretch before is done with
            for (int i = threadIdx.x; i < ((x1 - x0 + kMomGroup - 1) & -kMomGroup); i += 32 * kMomWarps) {
                const double X = (double)(2ll * (x0 + i) + 1) - P.org[0];
                double p = X, pe = 0.0;
#pragma unroll
                for (int a = 0; a < LMAX; ++a) {
                    pw[a * ch + i] = __dadd_rn(p, pe);
                    dd_power(p, pe, X);
                }
            }
            __syncthreads();
        }
        const long long tasks = (long long)((x1 - x0 + P.seg - 1) / P.seg) * jt * kt;
        long long t = w * tasks / W;
        const long long t1 = (w + 1) * tasks / W;
        while (t < t1) {
            const long long part = t / kt;  // segment and rows
            const int k0 = (int)(t - part * kt), k1 = (int)(t1 - t < kt - k0 ? k0 + (t1 - t) : kt);
            t += k1 - k0;
            const int s0 = x0 + (int)(part / jt) * P.seg, s1 = s0 + P.seg < x1 ? s0 + P.seg : x1;
            const int j = (int)(part % jt) * 32 + dj;
            double As[LMAX + 1][LMAX + 1], Ae[LMAX + 1][LMAX + 1];  // [a][c], a + c <= LMAX
#pragma unroll
            for (int a = 0; a <= LMAX; ++a)
#pragma unroll
                for (int c = 0; c <= LMAX; ++c) As[a][c] = Ae[a][c] = 0.0;
            for (int kk = k0; kk < k1; ++kk) {
                const int k = kk * nk + dk;
                const bool mine = j < P.ny && dk < nk && k < P.nz;
                const T* row = rho + (mine ? (long long)k * P.ny + j : 0ll) * P.nx;
                const int hi = mine ? s1 : 0;
                double Ts[LMAX + 1], Te[LMAX + 1];
#pragma unroll
                for (int a = 0; a <= LMAX; ++a) Ts[a] = Te[a] = 0.0;
                T nv[kMomGroup];  // the next group's cells: in flight while this one is worked on
                mom_load(row, s0, hi, vec, nv);
                for (int i = s0; i < s1; i += kMomGroup) {
                    T v[kMomGroup];
#pragma unroll
                    for (int e = 0; e < kMomGroup; ++e) v[e] = nv[e];
                    if (i + kMomGroup < s1) mom_load(row, i + kMomGroup, hi, vec, nv);
                    bool any = false;
#pragma unroll
                    for (int e = 0; e < kMomGroup; ++e) any = any || nonzero(v[e]);
                    if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
                    for (int g = 0; g < kMomGroup; g += kMomSum) {
                        double c[kMomSum];
#pragma unroll
                        for (int e = 0; e < kMomSum; ++e) c[e] = widen(v[g + e]);
#pragma unroll
                        for (int a = 0; a <= LMAX; ++a) {
                            double s;
                            if (a == 0) {
                                s = __dadd_rn(__dadd_rn(__dadd_rn(Te[a], c[0]), c[1]), __dadd_rn(c[2], c[3]));
                            } else {
                                const double2* p = reinterpret_cast<const double2*>(pw + (a - 1) * ch + (i - x0 + g));
                                const double2 pa = p[0], pb = p[1];
                                s = __fma_rn(c[3], pb.y, __fma_rn(c[2], pb.x, __fma_rn(c[1], pa.y, __fma_rn(c[0], pa.x, Te[a]))));
                            }
                            Te[a] = sum_error(Ts[a], s);  // goes into the next four cells' sum
                        }
                    }
                }
                const double Z = (double)(2ll * k + 1) - P.org[2];
                double zc = 1.0, ze = 0.0;
#pragma unroll
                for (int c = 0; c <= LMAX; ++c) {
#pragma unroll
                    for (int a = 0; a + c <= LMAX; ++a) dd_fma(As[a][c], Ae[a][c], Ts[a], Te[a], zc, ze);
                    dd_power(zc, ze, Z);
                }
            }
            // times Y^b, summed over the warp's rows: each step halves the lanes a moment is spread over and the moments a
            // lane holds, so lane n ends with moment n of the batch
            if constexpr (NM == 1) {
                dd_warp(As[0][0], Ae[0][0]);
                if (lane == 0) dd_merge(wm[warp][0][0], wm[warp][0][1], As[0][0], Ae[0][0]);
                continue;
            }
            const double Y = (double)(2ll * j + 1) - P.org[1];
            double yb[LMAX + 1], ye[LMAX + 1];
            yb[0] = 1.0, ye[0] = 0.0;
#pragma unroll
            for (int b = 1; b <= LMAX; ++b) {
                yb[b] = yb[b - 1], ye[b] = ye[b - 1];
                dd_power(yb[b], ye[b], Y);
            }
#pragma unroll
            for (int B = 0; B < NB; ++B) {
                double vs[32], ve[32];
#pragma unroll
                for (int n = 0; n < 32; ++n) vs[n] = ve[n] = 0.0;
#pragma unroll
                for (int l = 0; l <= LMAX; ++l)
#pragma unroll
                    for (int c = 0; c <= l; ++c)
#pragma unroll
                        for (int b = 0; b + c <= l; ++b) {
                            const int n = mono_off(l) + mono_at(l, b, c) - 32 * B;
                            if (n >= 0 && n < 32) dd_fma(vs[n], ve[n], As[l - b - c][c], Ae[l - b - c][c], yb[b], ye[b]);
                        }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const bool up = lane & o;
#pragma unroll
                    for (int n = 0; n < o; ++n) {
                        const double s2 = __shfl_xor_sync(0xffffffffu, up ? vs[n] : vs[n + o], o);
                        const double e2 = __shfl_xor_sync(0xffffffffu, up ? ve[n] : ve[n + o], o);
                        if (up) {
                            vs[n] = vs[n + o];
                            ve[n] = ve[n + o];
                        }
                        dd_merge(vs[n], ve[n], s2, e2);
                    }
                }
                dd_merge(wm[warp][32 * B + lane][0], wm[warp][32 * B + lane][1], vs[0], ve[0]);
            }
        }
    }
    __syncthreads();
    for (int m = threadIdx.x; m < NM; m += 32 * kMomWarps) {
        double s = wm[0][m][0], e = wm[0][m][1];
        for (int v = 1; v < kMomWarps; ++v) dd_merge(s, e, wm[v][m][0], wm[v][m][1]);
        tot[m][0] = s;
        tot[m][1] = e;
    }
    __syncthreads();
    if (!P.centred) {  // about the half cell -> about the origin, one axis after the other (binomials)
        for (int axis = 0; axis < 3; ++axis) {
            for (int m = threadIdx.x; m < NM; m += 32 * kMomWarps) {
                int l = 0, b = m, c = 0;
                while (mono_off(l + 1) <= m) ++l;
                for (b = m - mono_off(l); b > l - c; ++c) b -= l - c + 1;
                const int pw = axis == 0 ? l - b - c : axis == 1 ? b : c;  // the power of this axis
                double s = 0.0, e = 0.0, f = 1.0, fe = 0.0;               // binomial(pw, r) offset^r
                for (int r = 0; r <= pw; ++r) {
                    const int n = mono_off(l - r) + mono_at(l - r, b - (axis == 1 ? r : 0), c - (axis == 2 ? r : 0));
                    dd_fma(s, e, tot[n][0], tot[n][1], f, fe);
                    double g = 0.0, ge = 0.0;
                    dd_fma(g, ge, f, fe, P.off[axis][0], P.off[axis][1]);
                    const double n1 = (double)(pw - r), d = (double)(r + 1), gn = __dmul_rn(g, n1);
                    f = __ddiv_rn(gn, d);
                    fe = __ddiv_rn(__fma_rn(-f, d, gn) + __fma_rn(ge, n1, __fma_rn(g, n1, -gn)), d);
                }
                moved[m][0] = s;
                moved[m][1] = e;
            }
            __syncthreads();
            for (int m = threadIdx.x; m < NM; m += 32 * kMomWarps) {
                tot[m][0] = moved[m][0];
                tot[m][1] = moved[m][1];
            }
            __syncthreads();
        }
    }
    for (int q = threadIdx.x; q < NQ; q += 32 * kMomWarps) {
        int l = 0;
        while ((l + 1) * (l + 1) <= q) ++l;
        const int m = q - l * l - l;
        double s = 0.0, e = 0.0;
        for (int n = 0; n < (l + 1) * (l + 2) / 2; ++n) {
            const double c = kHarmonics.c[q][n];
            if (c != 0.0) dd_fma(s, e, tot[mono_off(l) + n][0], tot[mono_off(l) + n][1], c);
        }
        double vs = 0.0, ve = 0.0, us = 0.0, ue = 0.0, qs = 0.0, qe = 0.0;
        dd_fma(vs, ve, s, e, P.hl[l][0], P.hl[l][1]);
        dd_fma(us, ue, vs, ve, P.h3[0], P.h3[1]);
        dd_fma(qs, qe, us, ue, N.n[l * l + l + (m < 0 ? -m : m)]);
        partial[2 * ((long long)blockIdx.x * NQ + q)] = qs;
        partial[2 * ((long long)blockIdx.x * NQ + q) + 1] = qe;
    }
}

// one warp per moment: the pairs partial[2 (b nq + q) + {0, 1}] over the blocks b in a fixed order; out[q] = the
// rounded pair (one block over all moments took 166 us at lmax = 4, a serial chain of FP64 latencies; this 5)
__global__ void __launch_bounds__(32) k_finish_moments(const double* __restrict__ partial, int nq, double* __restrict__ out) {
    double s = 0.0, e = 0.0;
    for (int b = threadIdx.x; b < kMomBlocks; b += 32)
        dd_merge(s, e, partial[2 * ((long long)b * nq + blockIdx.x)], partial[2 * ((long long)b * nq + blockIdx.x) + 1]);
    dd_warp(s, e);
    if (threadIdx.x == 0) out[blockIdx.x] = s;
}

// Cells of a row in one task: whole rows where those make a task for every warp, else equal parts of at least 128 cells (with
// 64, 128^3 paid 133 us for a second Y^b and warp reduction against 117).  Float density, a call, us, for harmonics per cell
// (whose threads do not care about the shape), whole rows of one plane per task, and this: lmax 0: 512 x 4 x 512 45, 84, 35;
// 1024 x 1 x 1024 45, 207, 36; 2100 x 5 x 300 90, 272, 52; lmax 4: 900, 294, 110; 901, 778, 113; 2047, 991, 215.  Cubes from 224^3 on
// have enough rows and are as they were.
inline int mom_segment(int nx, int ny, int nz) {
    const long long nk = ny < 32 ? 32 / ny : 1, rows = ((nz + nk - 1) / nk) * ((ny + 31) / 32), all = kMomBlocks * kMomWarps;
    const long long parts = rows >= all ? 1 : all / rows;
    const long long len = (nx + parts - 1) / parts;
    return (int)((len > 128 ? len : 128) + kMomGroup - 1) & -kMomGroup;
}

// launch both kernels: the moments of rho (dense, device memory) into Q (device); scratch holds 2 kMomBlocks nq doubles
template <int LMAX>
cudaError_t launch_moments(const void* rho, int dtype, int nx, int ny, int nz, double h, const double* o, const YlmNorm& N,
                           double* scratch, double* Q, cudaStream_t st) {
    constexpr int NQ = (LMAX + 1) * (LMAX + 1);
    MomArgs P;
    P.nx = nx, P.ny = ny, P.nz = nz, P.seg = mom_segment(nx, ny, nz);
    const double h2 = h * h, h2e = fma(h, h, -h2);
    P.h3[0] = h2 * h;
    P.h3[1] = fma(h2, h, -P.h3[0]) + h2e * h;
    P.centred = 1;
    for (int a = 0; a < 3; ++a) {  // 2 o / h: the quotient and its rounding error, less the integer next to it (exact)
        const double q = 2.0 * o[a] / h;
        P.org[a] = -nearbyint(q);
        P.off[a][0] = q + P.org[a];
        P.off[a][1] = fma(-q, h, 2.0 * o[a]) / h;
        if (P.off[a][0] != 0.0 || P.off[a][1] != 0.0) P.centred = 0;
    }
    P.hl[0][0] = 1.0, P.hl[0][1] = 0.0;
    for (int l = 1; l <= kMaxL; ++l) {
        const double x = 0.25 * h, p = P.hl[l - 1][0] * x;
        P.hl[l][0] = p;
        P.hl[l][1] = fma(P.hl[l - 1][0], x, -p) + P.hl[l - 1][1] * x;
    }
    const int per16 = dtype == HG_DT_F64 ? 2 : 4;
    const bool vec = nx % per16 == 0 && (uintptr_t)rho % 16 == 0;
    const int th = 32 * kMomWarps;
    const int ch = nx < kMomStretch ? (nx + kMomGroup - 1) & -kMomGroup : kMomStretch;
    const int smem = LMAX * ch * (int)sizeof(double);
    constexpr int NM = mono_off(LMAX + 1), held = 16 * (kMomWarps * ((NM + 31) / 32) * 32 + 2 * NM);  // static part
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto* kernel, const auto* r) {
        // above 48 KB a kernel has to ask: each time, as a device reset forgets it, and always for the most, as another host
        // thread may be about to launch it for longer rows
        if (held + smem > 48 * 1024)
            e = cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     LMAX * kMomStretch * (int)sizeof(double));
        if (e != cudaSuccess) return;
        kernel<<<kMomBlocks, th, smem, st>>>(r, vec, P, N, scratch, ch);
        e = cudaGetLastError();
    };
    if (dtype == HG_DT_F64)
        launch(k_moments<double, LMAX>, (const double*)rho);
    else
        launch(k_moments<float, LMAX>, (const float*)rho);
    if (e != cudaSuccess) return e;
    k_finish_moments<<<NQ, 32, 0, st>>>(scratch, NQ, Q);
    return cudaGetLastError();
}

}  // namespace hg
