// Pieces of the compensated-float sub-step shared by the TMA-staged sweep (stencil_tma.cu, also the batched launch) and
// the flat sweep (sweep_flat.cuh): a lane's 4-cell group update, its stores, and the periodic ghosts of the
// new level.  Both sweeps thereby compute and store bit-identical results.
#pragma once

#include "cell.cuh"
#include "faces.cuh"
#include "hg_internal.cuh"

namespace hg {

__device__ __forceinline__ float el(const float4& v, int e) { return e == 0 ? v.x : e == 1 ? v.y : e == 2 ? v.z : v.w; }
__device__ __forceinline__ void set(float4& v, int e, float x) {
    if (e == 0) v.x = x; else if (e == 1) v.y = x; else if (e == 2) v.z = x; else v.w = x;
}

// One lane's 4 consecutive cells i0..i0+3 of row j, plane k: c/lc the level-n values of the group, hl/ll and hr/lr
// its x neighbours (cells i0-1 and i0+4), hs/hn (ls/ln) the -y/+y rows, hm/hp (lm/lp) the -z/+z planes, d the
// increments, r the source.  Stores hi', lo' (coded), dlt' at padded index q (cells beyond nx are not stored) and,
// for periodic grids, the ghosts that copy these cells.
__device__ __forceinline__ void group_update_store(const Layout& L, const Bnd& B, float nu2, int i0, int j, int k,
                                                   long long q, const float4& hc, const float4& lc, float hl, float ll,
                                                   float hr, float lr, const float4& hs, const float4& hn,
                                                   const float4& ls, const float4& ln, const float4& hm,
                                                   const float4& hp, const float4& lm, const float4& lp,
                                                   const float4& d, const float4& r, float* __restrict__ hi_n,
                                                   lo_t* __restrict__ lo_n, float* __restrict__ dlt) {
    float4 ho, lo, dout;
    f32k_update4_scalar(hc, lc, hl, ll, hr, lr, hs, hn, hm, hp, ls, ln, lm, lp, d, r, nu2, ho, lo, dout);
    if (!idx_ok(q, 4, L.elems, B.err)) return;
    const uint2 code = lo_encode4(ho, lo);
    auto code1 = [&](int e) { return __ushort_as_half((unsigned short)((e < 2 ? code.x : code.y) >> (16 * (e & 1)))); };
    if (i0 + 3 < L.nx) {
        *reinterpret_cast<float4*>(hi_n + q) = ho;
        *reinterpret_cast<uint2*>(lo_n + q) = code;
        *reinterpret_cast<float4*>(dlt + q) = dout;
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (i0 + e < L.nx) {
                hi_n[q + e] = el(ho, e);
                lo_n[q + e] = code1(e);
                dlt[q + e] = el(dout, e);
            }
    }
    if (B.periodic) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            periodic_x_ghosts(L, i0 + e, q + e, [&](long long g) {
                if (!idx_ok(g, 1, L.elems, B.err)) return;
                hi_n[g] = el(ho, e);
                lo_n[g] = code1(e);
            });
        periodic_yz_ghosts(L, j, k, q, [&](long long g) {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (i0 + e < L.nx && idx_ok(g + e, 1, L.elems, B.err)) {
                    hi_n[g + e] = el(ho, e);
                    lo_n[g + e] = code1(e);
                }
        });
    }
}

}  // namespace hg
