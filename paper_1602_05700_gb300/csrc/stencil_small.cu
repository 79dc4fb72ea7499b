// The sub-step of a small grid (arXiv 1602.05700, Sec. 1 Eq. HNeq., Sec. 2: k_g wave sub-steps per hydro step), where
// latency costs the time: the state sits in L2 and one sub-step is a few microseconds.
//
// A marching block (stencil_tma.cu, stencil.cu) pays its planes one after the other, and a small grid does not have
// enough blocks to hide that: 64^3 is 64 blocks of 8 planes, 14 us.  Here every group of cells (4 of a row for the
// compensated floats, 1 for FP64) is a thread of its own: all its neighbours are loaded at once, so a sub-step is one
// round of loads, one update and one round of stores.  Groups are numbered flat over rows and planes, so a 24-cell row
// leaves no lanes idle.  The Robin face ghosts of level n+1 depend on level n only and are further threads of the same
// launch (its first blocks, so that their longer chain starts first); periodic ghosts are stored with the cells they
// copy.  One launch per sub-step, by programmatic dependent launch: its blocks are resident, with their indices
// computed, when the previous sub-step ends.
//
// The adjoint's reverse sub-steps (ADJ) add level n to their running sum here, from the registers that hold it: a pass of
// its own took 32 us at 128^3 (float) beside the 9 us of the sub-step; this variant takes 12.
//
// Measured (Robin, us per sub-step, marching kernel with its own ghost launches -> this one):
//   compensated float  32^3 14.4 -> 2.5, 64^3 14.4 -> 3.7, 128^3 16.4 -> 9.0, 192^3 46.6 -> 38.5, 256^3 80.7 -> 88
//   FP64               32^3 21.2 -> 3.9, 64^3 18.0 -> 7.9, 128^3 39.6 -> 31.4, 192^3 139 -> 107, 256^3 228 -> 246
// Above the line (small_grid, stencil.cu) the z neighbours' re-reads (46 bytes of L2 traffic per cell against 30) cost
// more than the latency saved.  Blocks of 128 threads: 64 pay for block launches above 96^3, 256 and 512 wait longer
// for their slowest warp (64^3 f64: 7.9 against 8.4 and 9.5 us).  2 to 4 planes per thread were no faster anywhere
// (128^3: 9.4, 9.7 and 10.3 us): the loads they save hit L2, and they leave fewer threads to cover its latency.
#include "cell.cuh"
#include "faces.cuh"
#include "hg_internal.cuh"
#include "sweep_f32k.cuh"

namespace hg {

namespace {

constexpr int kSmallThreads = 128;

// group t of the flat numbering -> first cell i0, row j, plane k; false beyond the grid
__device__ __forceinline__ bool small_cell(const Layout& L, unsigned t, unsigned gpr, int width, int& i0, int& j, int& k) {
    const unsigned row = t / gpr;
    i0 = (int)(t - row * gpr) * width;
    k = (int)(row / (unsigned)L.ny);
    j = (int)(row - (unsigned)k * (unsigned)L.ny);
    return k < L.nz;
}

template <bool ADJ>
__global__ void __launch_bounds__(kSmallThreads) k_small_f32k(const SweepArgs A, unsigned gblocks, unsigned gpr,
                                                              float* acc_a, float* acc_b) {
    pdl_trigger();
    if (blockIdx.x < gblocks) {
        pdl_wait();
        robin_ghost(A, blockIdx.x * kSmallThreads + threadIdx.x);
        return;
    }
    const Layout& L = A.L;
    int i0, j, k;
    const bool mine = small_cell(L, (blockIdx.x - gblocks) * kSmallThreads + threadIdx.x, gpr, 4, i0, j, k);
    pdl_wait();
    if (!mine) return;
    const long long q = L.at(i0, j, k);
    // plain loads: with dependent launch the previous sub-step may still be writing when this kernel starts, so the
    // read-only path's premise does not hold
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
    group_update_store(L, A.B, A.nu2f, i0, j, k, q, hc, lc, hl, lo_decode(hl, cl), hr, lo_decode(hr, cr),
                       hs, hn, lo_decode4(hs, cs), lo_decode4(hn, cn), hm, hp, lo_decode4(hm, cm), lo_decode4(hp, cp), d,
                       r, (float*)A.hi_n, (lo_t*)A.lo_n, (float*)A.dlt);
}

template <bool ADJ>
__global__ void __launch_bounds__(kSmallThreads) k_small_f64(const SweepArgs A, unsigned gblocks, unsigned gpr, double* acc) {
    pdl_trigger();
    if (blockIdx.x < gblocks) {
        pdl_wait();
        robin_ghost(A, blockIdx.x * kSmallThreads + threadIdx.x);
        return;
    }
    const Layout& L = A.L;
    int i, j, k;
    const bool mine = small_cell(L, (blockIdx.x - gblocks) * kSmallThreads + threadIdx.x, gpr, 1, i, j, k);
    pdl_wait();
    if (!mine) return;
    const long long q = L.at(i, j, k);
    const double* p = (const double*)A.hi_c + q;
    double* o = (double*)A.hi_n;
    const double c = p[0];
    const double v = f64_update<false>(p[-1], p[1], p[-L.pitch], p[L.pitch], p[-L.plane], p[L.plane], c, o[q],
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

}  // namespace

// One sub-step cur -> 1 - cur of a small grid, all face ghosts included.  With acc_a the grid is an adjoint's shadow state
// (its source is zero and is not read) and level n is added to the running sum (acc_a, acc_b) on the way.
int launch_step_small(hg_grid* g, void* acc_a, void* acc_b) {
    const SweepArgs A = sweep_args(g, g->zb);
    const int width = g->prec == HG_PREC_F32K ? 4 : 1;
    const unsigned gpr = (unsigned)((g->nx + width - 1) / width);
    const unsigned groups = gpr * (unsigned)g->ny * (unsigned)g->nz;
    const unsigned gblocks = A.B.faces ? (unsigned)((A.B.off[6] + kSmallThreads - 1) / kSmallThreads) : 0u;
    const dim3 blocks(gblocks + (groups + kSmallThreads - 1) / kSmallThreads), threads(kSmallThreads);
    int rc = prof_begin(g);
    if (rc) return rc;
    if (width == 4)
        rc = launch_pdl(acc_a ? k_small_f32k<true> : k_small_f32k<false>, blocks, threads, 0, g->stream, A, gblocks, gpr,
                        (float*)acc_a, (float*)acc_b);
    else
        rc = launch_pdl(acc_a ? k_small_f64<true> : k_small_f64<false>, blocks, threads, 0, g->stream, A, gblocks, gpr,
                        (double*)acc_a);
    if (rc) return rc;
    HG_LAUNCHED("small-grid sub-step kernel");
    return prof_end(g);
}

}  // namespace hg
