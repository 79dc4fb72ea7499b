// One sub-step of the hyperbolic gravity equation (arXiv 1602.05700, Sec. 1 Eq. HNeq., Sec. 2):
//
//   phi^{n+1} = 2 phi^n - phi^{n-1} + nu^2 sum_{6 nb}(phi^n_nb - phi^n) - s,   s = (c_h dt)^2 4 pi G rho
//
// over the interior of the padded layout: which sweep a grid takes, the arguments of the sweeps, and the batched launches
// of many grids.  The sweeps are the flat one (sweep_flat.cuh, stencil_flat.cu) and, for large compensated-float grids, the
// TMA-staged one (sweep_tma.cuh, stencil_tma.cu).
//
// * f32k: float storage with compensated increments.  State per cell: hi + lo = phi^n (a float and its
//   rounding remainder, stored as a 16-bit code, cell.cuh) and dlt = phi^n - phi^{n-1}.  The sub-step is
//       dlt' = dlt + (nu^2 (L(hi) + L(lo)) - s),   (hi', lo') = hi + (lo + dlt')  by Fast2Sum,
//   so phi keeps ~36 bits: 24 bytes of HBM traffic per cell (read hi 4, lo 2, dlt 4, s 4; write hi' 4, lo' 2,
//   dlt' 4).  hi/lo ping-pong between two buffers (neighbours are read), dlt is updated in place.
// * f64: double storage, phi^{n+1} written over phi^{n-1}: 32 bytes per cell.  The update's 15 FP64 operations
//   (cell.cuh) run partly in integer instructions with the same bits (lap_int.cuh); GB300's FP64 rate and the
//   integer issue bound the kernel, not HBM.
// The stored "rho" array holds the scaled source s = (c_h dt)^2 4 pi G (rho - rho_bar).
#include "sweep_flat.cuh"
#include "sweep_tma.cuh"

namespace hg {

namespace {

constexpr int kWY = 8;

// z planes per block of the TMA-staged sweep: short chunks, many blocks -- the stage ring hides the z warm-up, and fine
// blocks balance the SMs, also where the last wave is nearly empty.  Us per sub-step (Robin) with 8 planes, the best of 6 to 48,
// and 25: 230^3 62.4, 62.3 (6), 83.1; 256^3 77.7, 76.8 (6), 92.1; 301x259x223 83.3, 83.2 (12), 91.8; 320^3 142.3, 141.5 (12), 152.2;
// 360^3 186.3, 186.3, 201.6; 400^3 264.2, 258.8 (12), 270.4; 512x256x128 73.5, 72.2 (6), 88.6; 512^3 497, 494 (6), 526.
int zchunk(const hg_grid* g) { return g->nz < 8 ? g->nz : 8; }

// entry of block b in a prefix table of n entries (first[0] = 0): 32 at a time, every lane one
__device__ __forceinline__ int batch_entry(const unsigned* __restrict__ first, int n, unsigned b) {
    int e = -1;
    for (int base = 0; base < n; base += 32) {
        const int i = base + (int)(threadIdx.x & 31);
        const unsigned m = __ballot_sync(0xffffffffu, i < n && __ldg(first + i) <= b);
        e += __popc(m);
        if (m != 0xffffffffu) break;
    }
    return e;
}

// The flat sweep of many grids: a block takes kBatchTiles tiles of one entry, whose arguments it copies to shared memory.
// With both precisions in the launch their blocks alternate in proportion to their numbers (share64 = blocks64 2^32 /
// blocks, rounded up: block b is the FP64 block number hi(b share64) where that number steps), so that FP64- and
// integer-bound blocks and HBM-bound ones are resident together all the way through.
template <bool F64, bool F32>
__global__ void __launch_bounds__(kBatchThreads, 8)
    k_batch_flat(const BatchEntry* __restrict__ tab64, const unsigned* __restrict__ first64, int n64,
                 const BatchEntry* __restrict__ tab32, const unsigned* __restrict__ first32, int n32, unsigned share64) {
    __shared__ SweepArgs A;
    __shared__ FlatGrid G;
    bool f64 = F64;
    unsigned b = blockIdx.x;
    if (F64 && F32) {
        const unsigned c = __umulhi(b, share64);
        f64 = __umulhi(b + 1, share64) > c;
        b = f64 ? c : b - c;
    }
    const unsigned* first = f64 ? first64 : first32;
    const int e = batch_entry(first, f64 ? n64 : n32, b);
    const BatchEntry& E = (f64 ? tab64 : tab32)[e];
    const unsigned tile0 = (b - __ldg(first + e)) * kBatchTiles;
    static_assert(sizeof(SweepArgs) % 4 == 0 && sizeof(FlatGrid) % 4 == 0, "copied by words");
    for (int w = threadIdx.x; w < (int)(sizeof(SweepArgs) / 4); w += kBatchThreads)
        ((unsigned*)&A)[w] = __ldg((const unsigned*)&E.A + w);
    if (threadIdx.x < sizeof(FlatGrid) / 4) ((unsigned*)&G)[threadIdx.x] = __ldg((const unsigned*)&E.G + threadIdx.x);
    __syncthreads();
    for (unsigned t = tile0; t < tile0 + kBatchTiles && t < G.tiles; ++t) {
        int i0, j, k;
        if (t < G.ghost_tiles) {
            robin_ghost(A, (int)(t * kBatchThreads + threadIdx.x));
            continue;
        }
        const int width = F64 && f64 ? 1 : 4;
        if (!(G.wide ? flat_cell<true>(A.L, G, t, width, i0, j, k) : flat_cell<false>(A.L, G, t, width, i0, j, k)))
            continue;
        if (F64 && f64)
            flat_f64<false>(A, i0, j, k, nullptr);
        else if (F32)
            flat_f32k<false>(A, i0, j, k, nullptr, nullptr);
    }
}

// Large float entries: the TMA-staged sweep with the single-grid kernel's launch shape (3 blocks per SM).  The tensor maps
// live in the table, in global memory; the issuing thread acquires them through the tensormap proxy before its first copy.
template <int WY, int S>
__global__ void __launch_bounds__(32 * (WY + 1), 3) k_batch_tma(const BatchEntry* __restrict__ tab,
                                                                const unsigned* __restrict__ first, int n) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long bars[2 * S];
    const int e = batch_entry(first, n, blockIdx.x);
    const BatchEntry& E = tab[e];
    const unsigned local = blockIdx.x - __ldg(first + e);
    const int bx = (int)(local % E.A.gx), by = (int)((local / E.A.gx) % E.A.gy), bz = (int)(local / (E.A.gx * E.A.gy));
    if (threadIdx.y == WY && threadIdx.x == 0)
        for (int m = 0; m < 4; ++m)
            asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(&E.m[m]) : "memory");
    tma_sweep<WY, S>(&E.m[0], &E.m[1], &E.m[2], &E.m[3], E.A, bx, by, bz, E.err, smem, bars);
}

}  // namespace

// Whether a grid's sub-steps run the flat sweep: always in FP64; float grids up to the size where the TMA-staged sweep
// overtakes it (cubes: 224^3 60.1 against 61.2 us, 192^3 38.0 against 45.6, 256^3 86 against 80).  A pinned block depth
// (hg_set_block_depth) asks for the TMA-staged sweep.
bool flat_sized(const hg_grid* g) {
    return g->prec == HG_PREC_F64 || (long long)g->nx * g->ny * g->nz <= 11500000LL;
}
bool flat_sweep(const hg_grid* g) { return flat_sized(g) && (g->prec == HG_PREC_F64 || g->zb == 0); }

// the sweep arguments of grid g for the sub-step cur -> 1 - cur, with z chunks of zb planes (0 = default rule)
SweepArgs sweep_args(const hg_grid* g, int zb) {
    SweepArgs A;
    const int nxt = 1 - g->cur;
    A.hi_c = g->phi[g->cur];
    A.lo_c = g->lo[g->cur];
    A.hi_n = g->phi[nxt];
    A.lo_n = g->lo[nxt];
    A.dlt = g->dlt[g->dcur];
    A.rho = g->rho;
    A.L = g->L;
    A.nu2 = g->nu2;
    A.nu2f = (float)g->nu2;
    A.zb = zb > 0 ? (zb < g->nz ? zb : g->nz) : zchunk(g);
    A.prec = g->prec;
    A.exact = g->texact;
    A.gx = (g->nx + 127) / 128;
    A.gy = (g->ny + kWY - 1) / kWY;
    A.B.faces = g->bc == HG_BC_ROBIN ? 1 : 0;
    A.B.periodic = g->bc == HG_BC_PERIODIC ? 1 : 0;
    A.B.zskip = g->ziface;
    A.B.err = g->derr;
    A.B.robin32 = g->robin32;
    A.B.robin = g->robin;
    for (int f = 0; f < 7; ++f) A.B.off[f] = g->F.off[f];
    return A;
}

unsigned sweep_blocks(const SweepArgs& A) { return A.gx * A.gy * (unsigned)((A.L.nz + A.zb - 1) / A.zb); }

// A single grid's sub-step, one launch with every face ghost of the new level in it: the flat sweep, or the TMA-staged
// sweep (Robin x/y faces by its producer warp, z faces by the first and last chunk); periodic ghosts are stored with
// the cells they copy.
int launch_step_single(hg_grid* g) {
    if (flat_sweep(g)) return launch_step_flat(g);
    const SweepArgs A = sweep_args(g, g->zb);
    int rc = prof_begin(g);
    if (rc) return rc;
    if ((rc = launch_sweep_f32k_tma(g, A))) return rc;
    return prof_end(g);
}

int launch_batch_flat(cudaStream_t st, const BatchEntry* tab64, const unsigned* first64, int n64, unsigned blocks64,
                      const BatchEntry* tab32, const unsigned* first32, int n32, unsigned blocks32) {
    const unsigned blocks = blocks64 + blocks32;
    if (!blocks) return HG_OK;
    const unsigned share64 = (unsigned)((((unsigned long long)blocks64 << 32) + blocks - 1) / blocks);
    if (!blocks32)
        k_batch_flat<true, false><<<blocks, kBatchThreads, 0, st>>>(tab64, first64, n64, tab32, first32, n32, 0u);
    else if (!blocks64)
        k_batch_flat<false, true><<<blocks, kBatchThreads, 0, st>>>(tab64, first64, n64, tab32, first32, n32, 0u);
    else
        k_batch_flat<true, true><<<blocks, kBatchThreads, 0, st>>>(tab64, first64, n64, tab32, first32, n32, share64);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? HG_OK : cuda_fail(e, "batched sub-step kernel");
}

int launch_batch_tma(cudaStream_t st, const BatchEntry* tab, const unsigned* first, int n, unsigned blocks) {
    if (!blocks) return HG_OK;
    static unsigned long long attr_done = 0;
    const int smem = kStages * StageGeom<kTmaWY>::bytes;
    int rc = smem_attr_once((const void*)k_batch_tma<kTmaWY, kStages>, smem, &attr_done);
    if (rc) return rc;
    k_batch_tma<kTmaWY, kStages><<<blocks, dim3(32, kTmaWY + 1), smem, st>>>(tab, first, n);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? HG_OK : cuda_fail(e, "batched TMA sub-step kernel");
}

}  // namespace hg
