// Field movement between the caller's dense arrays and the padded device layout, the gravitational acceleration
// -grad phi (arXiv 1602.05700: the force the hydro step consumes, Sec. 2), and the FP64 diagnostics of Sec. 4
// (Eq. error) and of the steady state (Eq. Poissoneq.).  Reductions are deterministic: fixed grid, per-block
// partial sums, one finishing block.
#include "cell.cuh"
#include "groups.cuh"
#include "hg_internal.cuh"

namespace hg {

static_assert(sizeof(lo_t) == sizeof(lo_code), "the compensation code is 16 bits wide");

namespace {

constexpr int kThreads = 256;
constexpr int kPackBlocks = 1216;  // 8 per SM; one partial sum each (fits the reduction scratch)

__device__ __forceinline__ void st(void* p, int dtype, long long i, double v) {
    if (dtype == HG_DT_F64)
        ((double*)p)[i] = v;
    else
        ((float*)p)[i] = (float)v;
}

// value of phi^n at padded index q, in double (F32K: float plus its decoded compensation)
__device__ __forceinline__ double phi_at(int prec, const void* p, const void* lo, long long q) {
    if (prec == HG_PREC_F64) return ((const double*)p)[q];
    return join_f32(((const float*)p)[q], ((const lo_t*)lo)[q]);
}

// visit every interior cell: blocks stride over the rows (j, k), threads over x (coalesced, no per-cell division)
template <class F>
__device__ __forceinline__ void for_cells(const Layout& L, F&& f) {
    const long long rows = (long long)L.ny * L.nz;
    for (long long row = blockIdx.x; row < rows; row += gridDim.x) {
        const int j = (int)(row % L.ny), k = (int)(row / L.ny);
        const long long base = row * L.nx;
        for (int i = threadIdx.x; i < L.nx; i += blockDim.x) f(i, j, k, base + i);
    }
}

// Source preparation: dst = scale * (src - shift) in the grid's layout and element type, where scale =
// (c dt)^2 4 pi G and shift = mean(rho) for periodic boundaries (MEAN; else nothing is subtracted).  Float input to a
// float grid is scaled in float (one rounding more than FP64, 6e-8 relative, and no slow FP64 instructions); every other
// combination in FP64, two operations per cell with the sum, which is what bounds it (256^3: 54 us of FP64 work; a
// subtraction of zero and a second look at the row made it 120).  With SUM the same pass also accumulates sum(src) for
// the FP64 mass: each thread in compensated float (TwoSum) or double, blocks in double, written as one partial per
// block (deterministic order).  The mean is one double in memory (written by the finishing kernel of the sum pass):
// dividing in every thread was 40 of the 46 us at 128^3.
__device__ __forceinline__ void two_sum_acc(float& s, float& c, float x) {
    const float t = s + x;
    const float bp = t - s;
    c += (s - (t - bp)) + (x - bp);
    s = t;
}

template <typename TS, typename TD, bool SUM, bool MEAN, int W, typename I>
__global__ void __launch_bounds__(kThreads) k_pack(const TS* __restrict__ src, TD* __restrict__ dst, Layout L,
                                                   const double* __restrict__ mean, double scale, double* partial) {
    pdl_trigger();
    float fs = 0.f, fc = 0.f;  // compensated float accumulator (float input)
    double ds = 0.0;           // double accumulator (double input)
    constexpr bool in_float = sizeof(TS) == 4 && sizeof(TD) == 4;
    const double shift = MEAN ? *mean : 0.0;
    const float scale32 = (float)scale, shift32 = (float)shift;
    for_groups<W, I>(L, [&](const Group<I>& g) {
        const Vec<TS, W> x = ldv<TS, W>(src + g.dense);
        Vec<TD, W> y;
#pragma unroll
        for (int e = 0; e < W; ++e) {
            if constexpr (in_float)
                y.v[e] = scale32 * (MEAN ? x.v[e] - shift32 : x.v[e]);
            else
                y.v[e] = (TD)(scale * (MEAN ? (double)x.v[e] - shift : (double)x.v[e]));
            if constexpr (SUM) {
                if constexpr (sizeof(TS) == 4)
                    two_sum_acc(fs, fc, x.v[e]);
                else
                    ds += x.v[e];
            }
        }
        stv<TD, W>(dst + L.at(g.i0, g.j, g.k), y);
    });
    if constexpr (SUM) {
        __shared__ double sh[32];
        const double v = block_sum(sizeof(TS) == 4 ? (double)fs + (double)fc : ds, sh);
        if (threadIdx.x == 0) partial[blockIdx.x] = v;
    }
}

// phi^n (interior) into a dense array.  A float result is the float nearest hi + lo, one float addition; a double one
// adds the two widened by integer instructions (widen, cell.cuh), one FP64 operation.  Through FP64 conversions this
// kernel took 963 us at 512^3.
template <typename TO, bool F64, int W, typename I>
__global__ void __launch_bounds__(kThreads) k_unpack(const void* p, const void* lo, TO* __restrict__ dst, Layout L) {
    pdl_trigger();
    pdl_wait();
    for_groups<W, I>(L, [&](const Group<I>& g) {
        const long long q = L.at(g.i0, g.j, g.k);
        Vec<TO, W> o;
        if constexpr (F64) {
            const Vec<double, W> x = ldv<double, W>((const double*)p + q);
#pragma unroll
            for (int e = 0; e < W; ++e) o.v[e] = (TO)x.v[e];
        } else {
            const Vec<float, W> h = ldv<float, W>((const float*)p + q);
            const Vec<lo_code, W> c = ldv<lo_code, W>((const lo_code*)lo + q);
#pragma unroll
            for (int e = 0; e < W; ++e) {
                const float l = lo_decode(h.v[e], __ushort_as_half(c.v[e]));
                if constexpr (sizeof(TO) == 4)
                    o.v[e] = __fadd_rn(h.v[e], l);
                else
                    o.v[e] = __dadd_rn(widen(h.v[e]), widen(l));
            }
        }
        stv<TO, W>(dst + g.dense, o);
    });
}

__global__ void k_unpack_ghosted(int prec, const void* p, const void* lo, double* dst, Layout L) {
    const int gx = L.nx + 2, gy = L.ny + 2, gz = L.nz + 2;
    const long long rows = (long long)gy * gz;
    for (long long row = blockIdx.x; row < rows; row += gridDim.x) {
        const int j = (int)(row % gy) - 1, k = (int)(row / gy) - 1;
        for (int ii = threadIdx.x; ii < gx; ii += blockDim.x) {
            const int i = ii - 1;
            const int out = (i < 0 || i >= L.nx) + (j < 0 || j >= L.ny) + (k < 0 || k >= L.nz);
            dst[row * gx + ii] = out > 1 ? 0.0 : phi_at(prec, p, lo, L.at(i, j, k));
        }
    }
}

// seed: level n from phi, level n-1 from prev (F64 into the two buffers; F32K: hi/lo split of phi and
// dlt = phi - prev rounded once).  Without prev the two levels are equal, so one split serves both; the split runs in
// integer instructions (split_f32): 375 us at 280^3 before, when each level took an FP64 subtraction and four conversions.
template <typename TS, bool F64, int W, typename I>
__global__ void __launch_bounds__(kThreads) k_seed(const TS* __restrict__ phi, const TS* __restrict__ prev, void* p_cur,
                                                   void* l_cur, void* p_oth, void* l_oth, void* dlt, Layout L) {
    for_groups<W, I>(L, [&](const Group<I>& g) {
        const long long q = L.at(g.i0, g.j, g.k);
        const Vec<TS, W> a = ldv<TS, W>(phi + g.dense);
        const Vec<TS, W> b = prev ? ldv<TS, W>(prev + g.dense) : a;
        if constexpr (F64) {
            Vec<double, W> x, y;
#pragma unroll
            for (int e = 0; e < W; ++e) {
                x.v[e] = (double)a.v[e];
                y.v[e] = (double)b.v[e];
            }
            stv<double, W>((double*)p_cur + q, x);
            stv<double, W>((double*)p_oth + q, y);
        } else {
            Vec<float, W> ha, hb, d;
            Vec<lo_code, W> la, lb;
#pragma unroll
            for (int e = 0; e < W; ++e) {
                lo_t l;
                if constexpr (sizeof(TS) == 4) {  // a float is its own split
                    ha.v[e] = a.v[e];
                    la.v[e] = 0;
                    hb.v[e] = b.v[e];
                    lb.v[e] = 0;
                    d.v[e] = __fsub_rn(a.v[e], b.v[e]);
                } else {
                    split_f32(a.v[e], ha.v[e], l);
                    la.v[e] = __half_as_ushort(l);
                    hb.v[e] = ha.v[e];
                    lb.v[e] = la.v[e];
                    d.v[e] = 0.f;
                    if (prev) {
                        split_f32(b.v[e], hb.v[e], l);
                        lb.v[e] = __half_as_ushort(l);
                        d.v[e] = (float)(a.v[e] - b.v[e]);
                    }
                }
            }
            stv<float, W>((float*)p_cur + q, ha);
            stv<lo_code, W>((lo_code*)l_cur + q, la);
            stv<float, W>((float*)p_oth + q, hb);
            stv<lo_code, W>((lo_code*)l_oth + q, lb);
            stv<float, W>((float*)dlt + q, d);
        }
    });
}

// a = -grad phi by central differences.  Compensated float grids with float output stay in float arithmetic
// ((hi+ - hi-) + (lo+ - lo-)); every other combination evaluates phi = hi + lo (or the double) in FP64.
__global__ void k_accel(int prec, const void* p, const void* lo, void* ax, void* ay, void* az, int ddt, Layout L,
                        double inv2h) {
    pdl_trigger();
    for_cells(L, [&](int i, int j, int k, long long c) {
        const long long q = L.at(i, j, k);
        if (prec == HG_PREC_F32K && ddt == HG_DT_F32) {
            const float* h = (const float*)p;
            const lo_t* lc = (const lo_t*)lo;
            auto l = [&](long long u) { return lo_decode(h[u], lc[u]); };
            const float s = (float)inv2h;
            ((float*)ax)[c] = -((h[q + 1] - h[q - 1]) + (l(q + 1) - l(q - 1))) * s;
            ((float*)ay)[c] = -((h[q + L.pitch] - h[q - L.pitch]) + (l(q + L.pitch) - l(q - L.pitch))) * s;
            ((float*)az)[c] = -((h[q + L.plane] - h[q - L.plane]) + (l(q + L.plane) - l(q - L.plane))) * s;
        } else {
            st(ax, ddt, c, -(phi_at(prec, p, lo, q + 1) - phi_at(prec, p, lo, q - 1)) * inv2h);
            st(ay, ddt, c, -(phi_at(prec, p, lo, q + L.pitch) - phi_at(prec, p, lo, q - L.pitch)) * inv2h);
            st(az, ddt, c, -(phi_at(prec, p, lo, q + L.plane) - phi_at(prec, p, lo, q - L.plane)) * inv2h);
        }
    });
}

// -grad phi of an FP64 grid in FP64: groups of W cells, each with its six neighbours (rows and planes out of L1 / L2),
// six FP64 operations per cell (the sign rides on the factor: (a - b)(-s) has the bits of -(a - b) s).  256^3: 162 us of
// FP64 work.
template <int W, typename I>
__global__ void __launch_bounds__(kThreads) k_accel_f64(const double* __restrict__ phi, double* __restrict__ ax,
                                                        double* __restrict__ ay, double* __restrict__ az, Layout L,
                                                        double inv2h) {
    pdl_trigger();
    const double s = -inv2h;
    for_groups<W, I>(L, [&](const Group<I>& g) {
        const double* p = phi + L.at(g.i0, g.j, g.k);
        const Vec<double, W> c = ldv<double, W>(p), ys = ldv<double, W>(p - L.pitch), yn = ldv<double, W>(p + L.pitch),
                             zm = ldv<double, W>(p - L.plane), zp = ldv<double, W>(p + L.plane);
        const double xl = p[-1], xr = p[W];
        Vec<double, W> x, y, z;
#pragma unroll
        for (int e = 0; e < W; ++e) {
            x.v[e] = ((e == W - 1 ? xr : c.v[(e + 1) % W]) - (e == 0 ? xl : c.v[(e + W - 1) % W])) * s;
            y.v[e] = (yn.v[e] - ys.v[e]) * s;
            z.v[e] = (zp.v[e] - zm.v[e]) * s;
        }
        stv<double, W>(ax + g.dense, x);
        stv<double, W>(ay + g.dense, y);
        stv<double, W>(az + g.dense, z);
    });
}

// Vectorised -grad phi for compensated float grids with float output (the per-hydro-step call): the work mapping
// of the sub-step kernel (a warp per 128-cell x-row, float4 per lane, x neighbours by shuffles, a z register queue)
// and the same arithmetic as k_accel.  HBM bytes per cell: read hi 4, lo 2; write ax, ay, az 12 = 18 B.  The kernel
// waits on its loads (no data reuse hides them), so four blocks per SM (64 registers) beat three (71 registers):
// 0.432 against 0.458 ms at 512^3.  Where the dense rows do not start on 16 bytes (nx not a multiple of 4) a lane's four
// results cannot be stored as one word, and element stores 16 bytes apart write every sector four times: the warp's row
// goes through shared memory instead and is stored 32 consecutive elements at a time.
constexpr int kAccWY = 8;
__global__ void __launch_bounds__(32 * kAccWY, 4) k_accel_f32k(const float* __restrict__ hi, const lo_t* __restrict__ lo,
                                                            float* __restrict__ ax, float* __restrict__ ay,
                                                            float* __restrict__ az, Layout L, float s, int zb) {
    __shared__ __align__(16) float row[kAccWY][128];
    pdl_trigger();
    const int lane = threadIdx.x;
    const int j = blockIdx.y * kAccWY + threadIdx.y;
    if (j >= L.ny) return;
    const int i0 = blockIdx.x * 128 + lane * 4;
    const bool active = i0 < L.nx, halo = i0 <= L.nx;
    const bool vec = (L.nx & 3) == 0;
    const int k0 = blockIdx.z * zb, k1 = min(L.nz, k0 + zb);
    auto ld4 = [](const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); };
    auto ldl4 = [](const lo_t* p) { return __ldg(reinterpret_cast<const uint2*>(p)); };
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    long long q = L.at(i0, j, k0);
    float4 hm = z4, hc = z4, lm = z4, lc = z4;
    if (halo) {
        hm = ld4(hi + q - L.plane);
        lm = lo_decode4(hm, ldl4(lo + q - L.plane));
        hc = ld4(hi + q);
        lc = lo_decode4(hc, ldl4(lo + q));
    }
    for (int k = k0; k < k1; ++k, q += L.plane) {
        float4 hp = z4, lp = z4, hs = z4, hn = z4, ls = z4, ln = z4;
        float hl = 0.f, hr = 0.f, ll = 0.f, lr = 0.f;
        if (halo) {
            hp = ld4(hi + q + L.plane);
            lp = lo_decode4(hp, ldl4(lo + q + L.plane));
        }
        if (active) {
            hs = ld4(hi + q - L.pitch);
            hn = ld4(hi + q + L.pitch);
            ls = lo_decode4(hs, ldl4(lo + q - L.pitch));
            ln = lo_decode4(hn, ldl4(lo + q + L.pitch));
            if (lane == 0) {
                hl = __ldg(hi + q - 1);
                ll = lo_decode(hl, lo[q - 1]);
            }
            if (lane == 31 && i0 + 4 <= L.nx) {
                hr = __ldg(hi + q + 4);
                lr = lo_decode(hr, lo[q + 4]);
            }
        }
        const float shl = __shfl_up_sync(0xffffffffu, hc.w, 1), sll = __shfl_up_sync(0xffffffffu, lc.w, 1);
        const float shr = __shfl_down_sync(0xffffffffu, hc.x, 1), slr = __shfl_down_sync(0xffffffffu, lc.x, 1);
        if (lane != 0) {
            hl = shl;
            ll = sll;
        }
        if (lane != 31) {
            hr = shr;
            lr = slr;
        }
        const float xh[6] = {hl, hc.x, hc.y, hc.z, hc.w, hr}, xl[6] = {ll, lc.x, lc.y, lc.z, lc.w, lr};
        const float hs_[4] = {hs.x, hs.y, hs.z, hs.w}, hn_[4] = {hn.x, hn.y, hn.z, hn.w};
        const float ls_[4] = {ls.x, ls.y, ls.z, ls.w}, ln_[4] = {ln.x, ln.y, ln.z, ln.w};
        const float hm_[4] = {hm.x, hm.y, hm.z, hm.w}, hp_[4] = {hp.x, hp.y, hp.z, hp.w};
        const float lm_[4] = {lm.x, lm.y, lm.z, lm.w}, lp_[4] = {lp.x, lp.y, lp.z, lp.w};
        float ox[4], oy[4], oz[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            ox[e] = -((xh[e + 2] - xh[e]) + (xl[e + 2] - xl[e])) * s;
            oy[e] = -((hn_[e] - hs_[e]) + (ln_[e] - ls_[e])) * s;
            oz[e] = -((hp_[e] - hm_[e]) + (lp_[e] - lm_[e])) * s;
        }
        const long long c = ((long long)k * L.ny + j) * L.nx + i0;
        auto store = [&](float* out, const float (&o)[4]) {
            if (vec) {
                if (active) *reinterpret_cast<float4*>(out + c) = make_float4(o[0], o[1], o[2], o[3]);
                return;
            }
            float* r = row[threadIdx.y];
            *reinterpret_cast<float4*>(r + 4 * lane) = make_float4(o[0], o[1], o[2], o[3]);
            __syncwarp();
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (i0 - 3 * lane + 32 * e < L.nx) out[c - 3 * lane + 32 * e] = r[lane + 32 * e];
            __syncwarp();
        };
        store(ax, ox);
        store(ay, oy);
        store(az, oz);
        hm = hc;
        hc = hp;
        lm = lc;
        lc = lp;
    }
}

// partial[b*NS + s] for the stats: 0 sum res^2, 1 max|res|, 2 sum (phi - phi_prev)^2, 3 sum phi^2, 4 max|phi|,
// 5 count of non-finite values
constexpr int NS = 6;
constexpr unsigned kStatsMax = (1u << 1) | (1u << 4);

__global__ void __launch_bounds__(kThreads) k_stats(int prec, const void* p, const void* lo, const void* pprev,
                                                    const void* dlt, const void* rho, Layout L, double ih2,
                                                    double inv_cdt2, double* partial) {
    __shared__ double sh[32];
    double a[NS] = {0, 0, 0, 0, 0, 0};
    for_cells(L, [&](int i, int j, int k, long long) {
        const long long q = L.at(i, j, k);
        const double pc = phi_at(prec, p, lo, q);
        double lap = 0.0;
        lap += phi_at(prec, p, lo, q - 1) - pc;
        lap += phi_at(prec, p, lo, q + 1) - pc;
        lap += phi_at(prec, p, lo, q - L.pitch) - pc;
        lap += phi_at(prec, p, lo, q + L.pitch) - pc;
        lap += phi_at(prec, p, lo, q - L.plane) - pc;
        lap += phi_at(prec, p, lo, q + L.plane) - pc;
        double r, d;
        if (prec == HG_PREC_F64) {
            r = ((const double*)rho)[q];
            d = pc - ((const double*)pprev)[q];
        } else {
            r = (double)((const float*)rho)[q];
            d = (double)((const float*)dlt)[q];
        }
        const double res = lap * ih2 - r * inv_cdt2;  // r = s = (c dt)^2 4 pi G (rho - rho_bar)
        a[0] += res * res;
        a[1] = fmax(a[1], fabs(res));
        a[2] += d * d;
        a[3] += pc * pc;
        a[4] = fmax(a[4], fabs(pc));
        if (!isfinite(pc) || !isfinite(d) || !isfinite(r)) a[5] += 1.0;
    });
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        double v = block_reduce(a[s], sh, (kStatsMax >> s) & 1u);
        if (threadIdx.x == 0) partial[(long long)blockIdx.x * NS + s] = v;
    }
}

// partial for compare: 0 sum (phi-P)^2, 1 sum P^2, 2 max|phi-P|, 3 max|P|, 4 sum ((phi-P)/P)^2
constexpr int NC = 5;
constexpr unsigned kCmpMax = (1u << 2) | (1u << 3);

__global__ void __launch_bounds__(kThreads) k_compare(int prec, const void* p, const void* lo, const double* P,
                                                      Layout L, double* partial) {
    __shared__ double sh[32];
    double a[NC] = {0, 0, 0, 0, 0};
    for_cells(L, [&](int i, int j, int k, long long c) {
        const double v = phi_at(prec, p, lo, L.at(i, j, k));
        const double b = P[c];
        const double d = v - b;
        a[0] += d * d;
        a[1] += b * b;
        a[2] = fmax(a[2], fabs(d));
        a[3] = fmax(a[3], fabs(b));
        a[4] += (d / b) * (d / b);
    });
#pragma unroll
    for (int s = 0; s < NC; ++s) {
        double v = block_reduce(a[s], sh, (kCmpMax >> s) & 1u);
        if (threadIdx.x == 0) partial[(long long)blockIdx.x * NC + s] = v;
    }
}

__global__ void __launch_bounds__(kThreads) k_sum(const void* src, int dt, long long n, double* partial) {
    __shared__ double sh[32];
    double a = 0.0;
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
    if (dt == HG_DT_F32) {
        const float* p = (const float*)src;
        float fs = 0.f, fc = 0.f;  // TwoSum-compensated float accumulation, then double
        const long long n4 = ((uintptr_t)p & 15) == 0 ? n >> 2 : 0;
        for (long long c = tid; c < n4; c += nt) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(p) + c);
            two_sum_acc(fs, fc, x.x);
            two_sum_acc(fs, fc, x.y);
            two_sum_acc(fs, fc, x.z);
            two_sum_acc(fs, fc, x.w);
        }
        for (long long c = 4 * n4 + tid; c < n; c += nt) two_sum_acc(fs, fc, p[c]);
        a = (double)fs + (double)fc;
    } else {
        const double* p = (const double*)src;
        for (long long c = tid; c < n; c += nt) a += p[c];
    }
    double v = block_sum(a, sh);
    if (threadIdx.x == 0) partial[blockIdx.x] = v;
}

// finish: out[s] = sum (or max, per bit of maxmask) over blocks of partial[b*ns + s], fixed order
// (with `mean`: *mean = out[0] / count)
__global__ void __launch_bounds__(kThreads) k_finish_mixed(const double* partial, int nblocks, int ns,
                                                           unsigned maxmask, double* out, double* mean = nullptr,
                                                           double count = 1.0) {
    __shared__ double sh[32];
    pdl_trigger();
    pdl_wait();
    for (int s = 0; s < ns; ++s) {
        const bool is_max = (maxmask >> s) & 1u;
        double v = 0.0;
        for (int b = threadIdx.x; b < nblocks; b += blockDim.x) {
            double x = partial[(long long)b * ns + s];
            v = is_max ? fmax(v, x) : v + x;
        }
        v = block_reduce(v, sh, is_max);
        if (threadIdx.x == 0) out[s] = v;
        if (mean && threadIdx.x == 0) *mean = v / count;
    }
}

// one block per row up to a cap (rows are strided by the grid)
inline unsigned cells_blocks(const hg_grid* g) {
    long long rows = (long long)(g->ny + 2) * (g->nz + 2);
    return (unsigned)(rows < 152 * 64 ? rows : 152 * 64);
}

}  // namespace

template <typename TS, typename TD, bool SUM, bool MEAN>
static void pack_launch(hg_grid* g, const void* src) {
    // the wider of the two types sets the group: 16 bytes of it
    using T = std::conditional_t<(sizeof(TS) < sizeof(TD)), TD, TS>;
    dispatch_groups<T>(g->L, dense_width<T>(g->L, {src}), [&](auto W, auto I) {
        const unsigned blocks = SUM ? (unsigned)kPackBlocks : group_blocks(g->L, W);
        k_pack<TS, TD, SUM, MEAN, W.value, decltype(I)><<<blocks, kThreads, 0, g->stream>>>(
            (const TS*)src, (TD*)g->rho, g->L, g->dmean, g->src, g->red);
    });
}

template <bool SUM, bool MEAN>
static int launch_pack(hg_grid* g, const void* src, int dtype) {
    if (dtype == HG_DT_F32 && g->prec == HG_PREC_F32K)
        pack_launch<float, float, SUM, MEAN>(g, src);
    else if (dtype == HG_DT_F32)
        pack_launch<float, double, SUM, MEAN>(g, src);
    else if (g->prec == HG_PREC_F32K)
        pack_launch<double, float, SUM, MEAN>(g, src);
    else
        pack_launch<double, double, SUM, MEAN>(g, src);
    HG_LAUNCHED("source preparation kernel");
    return HG_OK;
}

// Store the scaled source s = (c dt)^2 4 pi G (rho - rho_bar) and leave sum(rho) (FP64-accurate) in g->dsum on the
// device; nothing here waits for the GPU.  Periodic boundaries need the mean before scaling: a sum pass, then the
// pack reading the sum from device memory; otherwise one fused pass.
int prepare_source(hg_grid* g, const void* src, int dtype) {
    int rc;
    g->mass_pending = 1;
    if (g->bc == HG_BC_PERIODIC) {
        if ((rc = reduce_sum(g, src, dtype, g->dsum))) return rc;
        return launch_pack<false, true>(g, src, dtype);
    }
    if ((rc = launch_pack<true, false>(g, src, dtype))) return rc;
    // a dependent launch, as the sub-step behind it and k_unpack behind the acceleration are: of a whole 64^3 pass (density,
    // 20 sub-steps, acceleration, potential) 99.8 -> 96.0 us, of a periodic 128^3 one 218 -> 215
    if ((rc = launch_pdl(k_finish_mixed, dim3(1), dim3(kThreads), 0, g->stream, g->red, kPackBlocks, 1, 0u, g->dsum,
                         (double*)nullptr, 1.0)))
        return rc;
    HG_LAUNCHED("sum finish kernel");
    return HG_OK;
}

// Bring the mass and mean density of the last hg_set_density to the host (waits for the stream once per density)
int sync_mass(hg_grid* g) {
    if (!g->mass_pending) return HG_OK;
    double sum = 0.0;
    HG_CUDA(cudaMemcpyAsync(&sum, g->dsum, sizeof(double), cudaMemcpyDeviceToHost, g->stream));
    HG_CUDA(cudaStreamSynchronize(g->stream));
    g->mass = sum * g->h * g->h * g->h;
    g->rho_bar = g->bc == HG_BC_PERIODIC ? sum / ((double)g->nx * g->ny * g->nz) : 0.0;
    g->mass_pending = 0;
    return HG_OK;
}

int unpack_phi(hg_grid* g, void* dst, int dtype) {
    const void *p = g->phi[g->cur], *lo = g->lo[g->cur];
    int rc = HG_OK;
    auto run = [&](auto out, auto f64) {
        using TO = decltype(out);
        dispatch_groups<TO>(g->L, dense_width<TO>(g->L, {dst}), [&](auto W, auto I) {
            rc = launch_pdl(k_unpack<TO, f64.value, W.value, decltype(I)>, dim3(group_blocks(g->L, W)), dim3(kThreads), 0,
                            g->stream, p, lo, (TO*)dst, g->L);
        });
    };
    const bool f64 = g->prec == HG_PREC_F64;
    if (dtype == HG_DT_F64)
        f64 ? run(0.0, std::true_type()) : run(0.0, std::false_type());
    else
        f64 ? run(0.f, std::true_type()) : run(0.f, std::false_type());
    if (rc) return rc;
    HG_LAUNCHED("unpack kernel");
    return HG_OK;
}

int unpack_phi_ghosted(hg_grid* g, double* dst) {
    k_unpack_ghosted<<<cells_blocks(g), kThreads, 0, g->stream>>>(g->prec, g->phi[g->cur], g->lo[g->cur], dst, g->L);
    HG_LAUNCHED("ghosted unpack kernel");
    return HG_OK;
}

int set_phi_device(hg_grid* g, const void* phi, const void* prev, int dtype) {
    int oth = 1 - g->cur;
    auto run = [&](auto in, auto f64) {
        using TS = decltype(in);
        dispatch_groups<TS>(g->L, dense_width<TS>(g->L, {phi, prev}), [&](auto W, auto I) {
            k_seed<TS, f64.value, W.value, decltype(I)><<<group_blocks(g->L, W), kThreads, 0, g->stream>>>(
                (const TS*)phi, (const TS*)prev, g->phi[g->cur], g->lo[g->cur], g->phi[oth], g->lo[oth],
                g->dlt[g->dcur], g->L);
        });
    };
    const bool f64 = g->prec == HG_PREC_F64;
    if (dtype == HG_DT_F64)
        f64 ? run(0.0, std::true_type()) : run(0.0, std::false_type());
    else
        f64 ? run(0.f, std::true_type()) : run(0.f, std::false_type());
    HG_LAUNCHED("seed kernel");
    return HG_OK;
}

int accel(hg_grid* g, void* ax, void* ay, void* az, int dtype) {
    const bool aligned = ((uintptr_t)ax | (uintptr_t)ay | (uintptr_t)az) % 16 == 0;
    if (g->prec == HG_PREC_F32K && dtype == HG_DT_F32 && aligned) {
        const int zb = g->nz < 8 ? g->nz : 8;  // short z chunks: more blocks in flight (measured 0.459 ms at 512^3
                                                // against 0.489 ms with 32-plane chunks)
        dim3 block(32, kAccWY), grid((g->nx + 127) / 128, (g->ny + kAccWY - 1) / kAccWY, (g->nz + zb - 1) / zb);
        k_accel_f32k<<<grid, block, 0, g->stream>>>((const float*)g->phi[g->cur], (const lo_t*)g->lo[g->cur],
                                                    (float*)ax, (float*)ay, (float*)az, g->L,
                                                    (float)(1.0 / (2.0 * g->h)), zb);
    } else if (g->prec == HG_PREC_F64 && dtype == HG_DT_F64) {
        dispatch_groups<double>(g->L, dense_width<double>(g->L, {ax, ay, az}), [&](auto W, auto I) {
            k_accel_f64<W.value, decltype(I)><<<group_blocks(g->L, W), kThreads, 0, g->stream>>>(
                (const double*)g->phi[g->cur], (double*)ax, (double*)ay, (double*)az, g->L, 1.0 / (2.0 * g->h));
        });
    } else {
        k_accel<<<cells_blocks(g), kThreads, 0, g->stream>>>(g->prec, g->phi[g->cur], g->lo[g->cur], ax, ay, az,
                                                             dtype, g->L, 1.0 / (2.0 * g->h));
    }
    HG_LAUNCHED("acceleration kernel");
    return HG_OK;
}

int stats(hg_grid* g, hg_stats* s) {
    int rc = sync_mass(g);
    if (rc) return rc;
    if ((rc = device_error(g))) return rc;
    k_stats<<<kRedBlocks, kThreads, 0, g->stream>>>(g->prec, g->phi[g->cur], g->lo[g->cur], g->phi[1 - g->cur],
                                                    g->dlt[g->dcur], g->rho, g->L, 1.0 / (g->h * g->h),
                                                    1.0 / ((g->c * g->dt) * (g->c * g->dt)), g->red);
    HG_LAUNCHED("stats kernel");
    k_finish_mixed<<<1, kThreads, 0, g->stream>>>(g->red, kRedBlocks, NS, kStatsMax, g->dres);
    HG_LAUNCHED("stats finish kernel");
    double r[NS];
    HG_CUDA(cudaMemcpyAsync(r, g->dres, sizeof r, cudaMemcpyDeviceToHost, g->stream));
    HG_CUDA(cudaStreamSynchronize(g->stream));
    const double n = (double)g->nx * g->ny * g->nz;
    s->mass = g->mass;
    s->residual_rms = sqrt(r[0] / n);
    s->residual_max = r[1];
    s->change_rel = r[3] > 0.0 ? sqrt(r[2] / r[3]) : 0.0;
    s->phi_max = r[4];
    s->step = g->step;
    s->nonfinite = r[5] > 0.0 ? 1 : 0;
    return HG_OK;
}

int compare(hg_grid* g, const double* P, double out[3]) {
    k_compare<<<kRedBlocks, kThreads, 0, g->stream>>>(g->prec, g->phi[g->cur], g->lo[g->cur], P, g->L, g->red);
    HG_LAUNCHED("compare kernel");
    k_finish_mixed<<<1, kThreads, 0, g->stream>>>(g->red, kRedBlocks, NC, kCmpMax, g->dres);
    HG_LAUNCHED("compare finish kernel");
    double r[NC];
    HG_CUDA(cudaMemcpyAsync(r, g->dres, sizeof r, cudaMemcpyDeviceToHost, g->stream));
    HG_CUDA(cudaStreamSynchronize(g->stream));
    const double n = (double)g->nx * g->ny * g->nz;
    out[0] = sqrt(r[0] / r[1]);
    out[1] = r[2] / r[3];
    out[2] = sqrt(r[4] / n);
    return HG_OK;
}

int reduce_sum(hg_grid* g, const void* dense, int dtype, double* out_dev) {
    long long n = (long long)g->nx * g->ny * g->nz;
    k_sum<<<kPackBlocks, kThreads, 0, g->stream>>>(dense, dtype, n, g->red);
    HG_LAUNCHED("sum kernel");
    k_finish_mixed<<<1, kThreads, 0, g->stream>>>(g->red, kPackBlocks, 1, 0u, out_dev, g->dmean, (double)n);
    HG_LAUNCHED("sum finish kernel");
    return HG_OK;
}

}  // namespace hg
