// The flat sweep (sweep_flat.cuh) as a single grid's sub-step: one launch with every face ghost of the new level in it, by
// programmatic dependent launch, so its blocks are resident, with their indices computed, when the previous sub-step ends.
//
// Measured (Robin, us per sub-step, marching kernels with their own ghost launches -> this one):
//   compensated float  32^3 14.4 -> 2.4, 64^3 14.4 -> 3.5, 128^3 16.4 -> 8.4, 192^3 46.6 -> 38.0, 256^3 80.7 -> 86
//   FP64 (1/r field)   32^3 21.2 -> 3.2, 64^3 18.0 -> 5.7, 128^3 39.6 -> 20.6, 192^3 139 -> 67.4, 256^3 228 -> 155
// (the FP64 figures include the integer forms of lap_int.cuh, and two cells per thread from 600,000 cells).  Blocks of 128
// threads: 64 pay for block launches above 96^3, 256 and 512 wait longer for their slowest warp.  2 to 4 planes per thread
// were no faster anywhere (float 128^3: 9.4, 9.7 and 10.3 us against 9.0): the loads they save hit L2, and they leave fewer
// threads to cover its latency.
//
// The adjoint's reverse sub-steps (ADJ) add level n to their running sum from the registers that hold it: a pass of its own
// took 32 us at 128^3 (float) beside the 9 us of the sub-step; this variant takes 12.
#include <type_traits>

#include "sweep_flat.cuh"

namespace hg {

namespace {

constexpr int kFlatThreads = 128;

// FP64: two cells per thread from here on.  They share the conversions of the integer forms (194 instructions per cell
// instead of 248) and move 16 bytes per access; smaller grids want the threads.  Measured, us per sub-step, one -> two cells:
// 32^3 2.59 -> 4.1, 64^3 4.82 -> 4.82, 96^3 10.9 -> 10.5, 128^3 22.6 -> 20.6, 192^3 75.4 -> 67.4, 256^3 176 -> 155,
// 301x259x223 184 -> 165.  (Marching 2 to 16 planes per thread, with or without square tiles, 144-150 us in a field where this
// takes 148: the loads it saves do not bound it.)  The adjoint's reverse sub-steps keep one cell per thread: lambda changes sign, and
// a warp of 64 cells is oftener left to FP64.  Us per reverse sub-step, one -> two cells: 64 injected cells 96^3 29.0 -> 29.5, 128^3
// 61.0 -> 63.4, 192^3 180 -> 190, 256^3 370 -> 398; noise in every cell 30.5 -> 30.3, 68.2 -> 68.3, 223 -> 223, 523 -> 521; only a smooth
// injection of one sign gains, 12.6 -> 13.8, 25.2 -> 25.9, 90.6 -> 84.7, 209 -> 192.
constexpr long long kPairCells = 600000;

template <bool ADJ, bool WIDE>
__global__ void __launch_bounds__(kFlatThreads) k_step_f32k_flat(const SweepArgs A, const FlatGrid G, float* acc_a,
                                                                 float* acc_b) {
    pdl_trigger();
    if (blockIdx.x < G.ghost_tiles) {
        pdl_wait();
        robin_ghost(A, blockIdx.x * kFlatThreads + threadIdx.x);
        return;
    }
    int i0, j, k;
    const bool mine = flat_cell<WIDE>(A.L, G, blockIdx.x, 4, i0, j, k);
    pdl_wait();
    if (mine) flat_f32k<ADJ>(A, i0, j, k, acc_a, acc_b);
}

template <bool ADJ, bool WIDE>
__global__ void __launch_bounds__(kFlatThreads, 10) k_step_f64(const SweepArgs A, const FlatGrid G, double* acc) {
    pdl_trigger();
    if (blockIdx.x < G.ghost_tiles) {
        pdl_wait();
        robin_ghost(A, blockIdx.x * kFlatThreads + threadIdx.x);
        return;
    }
    int i, j, k;
    const bool mine = flat_cell<WIDE>(A.L, G, blockIdx.x, 1, i, j, k);
    pdl_wait();
    if (mine) flat_f64<ADJ>(A, i, j, k, acc);
}

// 7 resident blocks of 72 registers; 6 and 8 (spills) are both 3-8% slower
template <bool ODD, bool WIDE>
__global__ void __launch_bounds__(kFlatThreads, 7) k_step_f64x2(const SweepArgs A, const FlatGrid G) {
    pdl_trigger();
    if (blockIdx.x < G.ghost_tiles) {
        pdl_wait();
        robin_ghost(A, blockIdx.x * kFlatThreads + threadIdx.x);
        return;
    }
    int i, j, k;
    const bool mine = flat_cell<WIDE>(A.L, G, blockIdx.x, 2, i, j, k);
    pdl_wait();
    if (mine) flat_f64x2<ODD>(A, i, j, k);
}

}  // namespace

FlatGrid flat_grid(const hg_grid* g, int threads, int width) {
    const long long gpr = (g->nx + width - 1) / width, plane = gpr * g->ny;
    FlatGrid G;
    G.gpr = fast_div((unsigned)gpr);
    G.per_plane = fast_div((unsigned)((plane + threads - 1) / threads));
    G.wide = plane + threads >= (1LL << 31);
    G.ghost_tiles = g->bc == HG_BC_ROBIN ? (unsigned)((g->F.off[6] + threads - 1) / threads) : 0u;
    G.tiles = G.ghost_tiles + G.per_plane.d * (unsigned)g->nz;
    return G;
}

int launch_step_flat(hg_grid* g, void* acc_a, void* acc_b) {
    const SweepArgs A = sweep_args(g, 0);
    const bool pairs = g->prec == HG_PREC_F64 && !acc_a && (long long)g->nx * g->ny * g->nz >= kPairCells;
    const FlatGrid G = flat_grid(g, kFlatThreads, g->prec == HG_PREC_F32K ? 4 : pairs ? 2 : 1);
    int rc = prof_begin(g);
    if (rc) return rc;
    auto launch = [&](auto adj, auto wide) {
        if (g->prec == HG_PREC_F32K)
            return launch_pdl(k_step_f32k_flat<adj.value, wide.value>, dim3(G.tiles), dim3(kFlatThreads), 0, g->stream, A, G,
                              (float*)acc_a, (float*)acc_b);
        if (pairs)
            return launch_pdl(g->nx % 2 ? k_step_f64x2<true, wide.value> : k_step_f64x2<false, wide.value>, dim3(G.tiles),
                              dim3(kFlatThreads), 0, g->stream, A, G);
        return launch_pdl(k_step_f64<adj.value, wide.value>, dim3(G.tiles), dim3(kFlatThreads), 0, g->stream, A, G,
                          (double*)acc_a);
    };
    if (acc_a)
        rc = G.wide ? launch(std::true_type(), std::true_type()) : launch(std::true_type(), std::false_type());
    else
        rc = G.wide ? launch(std::false_type(), std::true_type()) : launch(std::false_type(), std::false_type());
    if (rc) return rc;
    HG_LAUNCHED("sub-step kernel");
    return prof_end(g);
}

}  // namespace hg
