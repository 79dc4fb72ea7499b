// The flat sweep: one sub-step (arXiv 1602.05700, Sec. 1 Eq. HNeq., Sec. 2: k_g wave sub-steps per hydro step) with a thread
// of its own for every group of cells (4 of a row for the compensated floats, 1 or 2 for FP64), no marching and no shared
// memory.  All FP64 sub-steps, those of float grids up to 224^3, the adjoint's and the batched launches run it
// (stencil_flat.cu, batch kernels in stencil.cu).
//
// A block that marches in z pays its planes one after the other and keeps few warps resident (the FP64 sweep it replaces:
// 108 registers, 16 warps per SM).  Here all neighbours of a group are loaded at once, a small grid is one round of
// loads, one update and one round of stores, and a large FP64 grid has 28 warps of 64 cells per SM to cover the latencies of the FP64
// and integer pipes that bound it.  The y and z neighbours are re-read through L1 and L2 (46 bytes of L2 traffic per float
// cell against 30 for the staged sweep, which is why large float grids keep that one).
//
// Groups are numbered flat over the rows of a plane, so a 24-cell row leaves no lanes idle.  A tile is one block's width
// of them: first the tiles of Robin ghosts (level n+1 of a ghost depends on level n only, so they run beside the
// interior, and first because their chain is longer), then those of each plane.  Periodic ghosts are stored with the
// cells they copy.
#pragma once

#include "cell.cuh"
#include "faces.cuh"
#include "hg_internal.cuh"
#include "sweep_f32k.cuh"

namespace hg {

// first cell i0, row j, plane k of this thread's group in a tile behind the ghost tiles; false beyond the plane.  WIDE: a
// plane of 2^31 groups or more
template <bool WIDE>
__device__ __forceinline__ bool flat_cell(const Layout& L, const FlatGrid& G, unsigned tile, int width, int& i0, int& j,
                                          int& k) {
    const unsigned b = tile - G.ghost_tiles;
    k = (int)G.per_plane.div(b);
    const unsigned in = b - (unsigned)k * G.per_plane.d;
    if (WIDE) {
        const long long t = (long long)in * blockDim.x + threadIdx.x, r = t / G.gpr.d;
        j = r < L.ny ? (int)r : L.ny;
        i0 = (int)(t - r * G.gpr.d) * width;
    } else {
        const unsigned t = in * blockDim.x + threadIdx.x;
        j = (int)G.gpr.div(t);
        i0 = (int)(t - (unsigned)j * G.gpr.d) * width;
    }
    return j < L.ny;
}

// One tile of a compensated-float grid.  Loads are plain: with dependent launch the previous sub-step may still be
// writing when the kernel starts, so the read-only path's premise does not hold.  ADJ: the grid is an adjoint's shadow
// state; its source is zero and not read, and level n is added to the running sum (acc_a, acc_b) on the way.
template <bool ADJ>
__device__ __forceinline__ void flat_f32k(const SweepArgs& A, int i0, int j, int k, float* acc_a, float* acc_b) {
    const Layout& L = A.L;
    const long long q = L.at(i0, j, k);
    const float* H = (const float*)A.hi_c + q;
    const lo_t* C = (const lo_t*)A.lo_c + q;
    auto h4 = [&](long long o) { return *reinterpret_cast<const float4*>(H + o); };
    auto c4 = [&](long long o) { return *reinterpret_cast<const uint2*>(C + o); };
    const float4 hc = h4(0), hs = h4(-L.pitch), hn = h4(L.pitch), hm = h4(-L.plane), hp = h4(L.plane);
    const uint2 cc = c4(0), cs = c4(-L.pitch), cn = c4(L.pitch), cm = c4(-L.plane), cp = c4(L.plane);
    const float hl = H[-1], hr = H[4];
    const lo_t cl = C[-1], cr = C[4];
    const float4 d = *reinterpret_cast<const float4*>((const float*)A.dlt + q);
    const float4 lc = lo_decode4(hc, cc);
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    if (ADJ) {
        float4 a = *reinterpret_cast<const float4*>(acc_a + q), b = *reinterpret_cast<const float4*>(acc_b + q);
        accumulate_f32k(a.x, b.x, hc.x, lc.x);
        accumulate_f32k(a.y, b.y, hc.y, lc.y);
        accumulate_f32k(a.z, b.z, hc.z, lc.z);
        accumulate_f32k(a.w, b.w, hc.w, lc.w);
        *reinterpret_cast<float4*>(acc_a + q) = a;  // beyond nx: the row's padding, as the loads
        *reinterpret_cast<float4*>(acc_b + q) = b;
    } else {
        r = *reinterpret_cast<const float4*>((const float*)A.rho + q);
    }
    group_update_store(L, A.B, A.nu2f, i0, j, k, q, hc, lc, hl, lo_decode(hl, cl), hr, lo_decode(hr, cr), hs, hn,
                       lo_decode4(hs, cs), lo_decode4(hn, cn), hm, hp, lo_decode4(hm, cm), lo_decode4(hp, cp), d, r,
                       (float*)A.hi_n, (lo_t*)A.lo_n, (float*)A.dlt);
}

// one cell of an FP64 grid
template <bool ADJ>
__device__ __forceinline__ void flat_f64(const SweepArgs& A, int i, int j, int k, double* acc) {
    const Layout& L = A.L;
    const long long q = L.at(i, j, k);
    const double* p = (const double*)A.hi_c + q;
    double* o = (double*)A.hi_n;
    const double c = p[0];
    const double v = f64_update(p[-1], p[1], p[-L.pitch], p[L.pitch], p[-L.plane], p[L.plane], c, o[q],
                                ADJ ? 0.0 : ((const double*)A.rho)[q], A.nu2);
    if (ADJ) acc[q] = __dadd_rn(acc[q], c);
    if (!idx_ok(q, 1, L.elems, A.B.err)) return;
    o[q] = v;
    if (A.B.periodic) {
        auto put = [&](long long gq) {
            if (idx_ok(gq, 1, L.elems, A.B.err)) o[gq] = v;
        };
        periodic_x_ghosts(L, i, q, put);
        periodic_yz_ghosts(L, j, k, q, put);
    }
}

// Two cells i, i+1 of an FP64 grid's row.  ODD: rows have an odd number of cells, and `two` is false for the last one, whose
// partner is the +x ghost (an instance of its own: the test costs even rows 1.5%)
template <bool ODD>
__device__ __forceinline__ void flat_f64x2(const SweepArgs& A, int i, int j, int k) {
    const Layout& L = A.L;
    const bool two = !ODD || i + 1 < L.nx;
    const long long q = L.at(i, j, k);
    const double* p = (const double*)A.hi_c + q;
    double* o = (double*)A.hi_n;
    auto d2 = [](const double* a) { return *reinterpret_cast<const double2*>(a); };  // rows start on 128 bytes, i is even
    const double2 cc = d2(p), ys = d2(p - L.pitch), yn = d2(p + L.pitch), zm = d2(p - L.plane), zp = d2(p + L.plane);
    const double2 rs = d2((const double*)A.rho + q);
    double pv[2];
    load_pair(o + q, two, pv);
    const double xl = p[-1], xr = p[two ? 2 : 1];
    double n[2][6] = {{xl, cc.y, ys.x, yn.x, zm.x, zp.x}, {cc.x, xr, ys.y, yn.y, zm.y, zp.y}};
    if (!two) {  // neighbours that leave the form of the first cell's sum as it is
#pragma unroll
        for (int e = 1; e < 6; ++e) n[1][e] = cc.y;
    }
    double v[2];
    f64_update2({cc.x, cc.y}, n, pv, {rs.x, rs.y}, A.nu2, v);
    if (!idx_ok(q, 2, L.elems, A.B.err)) return;
    if (two)
        *reinterpret_cast<double2*>(o + q) = make_double2(v[0], v[1]);
    else
        o[q] = v[0];
    if (A.B.periodic) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            if (e == 1 && !two) break;
            auto put = [&](long long gq) {
                if (idx_ok(gq, 1, L.elems, A.B.err)) o[gq] = v[e];
            };
            periodic_x_ghosts(L, i + e, q + e, put);
            periodic_yz_ghosts(L, j, k, q + e, put);
        }
    }
}

}  // namespace hg
