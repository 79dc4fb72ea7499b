// Face ghosts of one sub-step, shared by the sweeps: the Robin update of a single ghost (one thread each, from level n
// only, so it runs beside the interior in the same launch) and the periodic copies a sweep writes as it stores the
// cells next to a face (no second pass, no second launch).
#pragma once

#include "cell.cuh"
#include "hg_internal.cuh"

namespace hg {

// ghost t of the face-major enumeration -> padded indices of the ghost and of its interior neighbour
__device__ __forceinline__ void ghost_cells(const Layout& L, const Bnd& B, int t, long long& qg, long long& qi) {
    int f = 0, base = 0;
#pragma unroll
    for (int u = 1; u < 6; ++u)
        if (t >= (int)B.off[u]) {
            f = u;
            base = (int)B.off[u];
        }
    const int r = t - base;
    const int na = f < 2 ? L.ny : L.nx;
    const int b = r / na, a = r - b * na;
    switch (f) {
        case 0: qg = L.at(-1, a, b); qi = qg + 1; break;
        case 1: qg = L.at(L.nx, a, b); qi = qg - 1; break;
        case 2: qg = L.at(a, -1, b); qi = qg + L.pitch; break;
        case 3: qg = L.at(a, L.ny, b); qi = qg - L.pitch; break;
        case 4: qg = L.at(a, b, -1); qi = qg + L.plane; break;
        default: qg = L.at(a, b, L.nz); qi = qg - L.plane; break;
    }
}

// Robin ghost t of level n+1 (the sweep neither reads nor writes it)
__device__ __forceinline__ void robin_ghost(const SweepArgs& A, int t) {
    if (t >= (int)A.B.off[6]) return;
    if (((A.B.zskip & 1) && t >= (int)A.B.off[4] && t < (int)A.B.off[5]) || ((A.B.zskip & 2) && t >= (int)A.B.off[5]))
        return;  // a slab interface: the caller supplies that ghost plane
    long long qg, qi;
    ghost_cells(A.L, A.B, t, qg, qi);
    if (!idx_ok(qg, 1, A.L.elems, A.B.err)) return;
    if (A.prec == HG_PREC_F32K) {
        const float* hc = (const float*)A.hi_c;
        const lo_t* lc = (const lo_t*)A.lo_c;
        const float2 ab = A.B.robin32[t];
        const float hg = hc[qg], hi = hc[qi];
        float gh, gl;
        robin_update_f32k(ab.x, ab.y, hg, lo_decode(hg, lc[qg]), hi, lo_decode(hi, lc[qi]), gh, gl);
        ((float*)A.hi_n)[qg] = gh;
        ((lo_t*)A.lo_n)[qg] = lo_encode(gh, gl);
    } else {
        const double* pc = (const double*)A.hi_c;
        const double* R = A.B.robin;
        ((double*)A.hi_n)[qg] = robin_update_f64(R[3 * t], R[3 * t + 1], R[3 * t + 2], pc[qg], pc[qi]);
    }
}

// The periodic ghosts that copy cell (i, j, k) at padded index q: put(index) stores the cell's new value there.  Each
// ghost copies exactly one cell, so it is written once.
template <class Put>
__device__ __forceinline__ void periodic_x_ghosts(const Layout& L, int i, long long q, Put&& put) {
    if (i == 0) put(q + L.nx);
    if (i == L.nx - 1) put(q - L.nx);
}
template <class Put>
__device__ __forceinline__ void periodic_yz_ghosts(const Layout& L, int j, int k, long long q, Put&& put) {
    if (j == 0) put(q + L.ny * L.pitch);
    if (j == L.ny - 1) put(q - L.ny * L.pitch);
    if (k == 0) put(q + L.nz * L.plane);
    if (k == L.nz - 1) put(q - L.nz * L.plane);
}

}  // namespace hg
