// Discrete adjoint of the sub-stepping, for gradients dL/drho through T sub-steps (the differentiation workload;
// the paper itself has no adjoint: this is the transpose of its Eq. HNeq. time-stepper, Sec. 2).
//
// The sub-step is linear in (phi^n, phi^{n-1}, s).  Writing its transpose in gather form gives, for the adjoint
// variables lambda^m = dL/dphi^m (interior cells) and the Robin ghost variables,
//   lambda_c^m = 2 lambda_c^{m+1} - lambda_c^{m+2} + nu^2 sum_{6 nb}(mu_nb^{m+1} - lambda_c^{m+1}) + injection,
//   mu_g^m     = alpha_g mu_g^{m+1} + beta_g lambda_i^{m+1}                              (Robin ghosts),
// where mu_nb is lambda_nb for an interior neighbour, 0 for a Dirichlet ghost (boundary data do not depend on rho),
// the wrapped value for a periodic ghost, and mu_g = (beta_g / nu^2) dL/dphi_g for a Robin ghost.  With that scaling
// the recursion is exactly the forward sub-step with a zero source, so the adjoint runs on the same kernels, in a
// shadow grid of the same geometry, precision and boundary condition whose boundary data are zero.
// Then dL/ds_c = -sum_{m=1..T} lambda_c^m and dL/drho = (c dt)^2 4 pi G dL/ds (minus its mean for periodic
// boundaries, the transpose of rho -> rho - mean(rho)).  The recursion needs no forward states.
//
// Kernels here: add an injection into the shadow state, accumulate sum_m lambda^m (float pairs for the compensated
// precision, double for FP64), and turn the sum into the gradient.
#include "cell.cuh"
#include "groups.cuh"
#include "hg_internal.cuh"

namespace hg {

namespace {

constexpr int kThreads = 256;

// lambda^m += v on the interior; for the compensated state the increment dlt = lambda^m - lambda^{m+1} moves too.  A
// double enters as the float pair nearest to it.
template <typename T, bool F64, int W, typename I>
__global__ void __launch_bounds__(kThreads) k_inject(const T* __restrict__ v, void* hi, void* lo, void* dlt, Layout L) {
    for_groups<W, I>(L, [&](const Group<I>& g) {
        const long long q = L.at(g.i0, g.j, g.k);
        const Vec<T, W> x = ldv<T, W>(v + g.dense);
        if constexpr (F64) {
            Vec<double, W> p = ldv<double, W>((double*)hi + q);
#pragma unroll
            for (int e = 0; e < W; ++e) p.v[e] += (double)x.v[e];
            stv<double, W>((double*)hi + q, p);
        } else {
            Vec<float, W> h = ldv<float, W>((float*)hi + q), d = ldv<float, W>((float*)dlt + q);
            Vec<lo_code, W> c = ldv<lo_code, W>((lo_code*)lo + q);
#pragma unroll
            for (int e = 0; e < W; ++e) {
                const float xh = (float)x.v[e];
                const float xl = sizeof(T) == 4 ? 0.f : (float)((double)x.v[e] - (double)xh);
                float s, r;
                two_sum(h.v[e], xh, s, r);
                const float t = (lo_decode(h.v[e], __ushort_as_half(c.v[e])) + xl) + r;
                const float hn = s + t;
                h.v[e] = hn;
                c.v[e] = __half_as_ushort(lo_encode(hn, t - (hn - s)));
                d.v[e] += xh;
            }
            stv<float, W>((float*)hi + q, h);
            stv<lo_code, W>((lo_code*)lo + q, c);
            stv<float, W>((float*)dlt + q, d);
        }
    });
}

// acc += lambda^m on the interior, for the float grids whose sub-step does not do it on the way (flat_sweep, stencil.cu).
// All arrays are padded, so groups of 4 (rows have room for the last one) whatever nx is.
__global__ void __launch_bounds__(kThreads) k_accumulate(const float* __restrict__ hi, const lo_code* __restrict__ lo,
                                                         float* __restrict__ acc_a, float* __restrict__ acc_b, Layout L,
                                                         unsigned gpr) {
    for (long long t = blockIdx.x * (long long)kThreads + threadIdx.x; t < (long long)gpr * L.ny * L.nz;
         t += (long long)gridDim.x * kThreads) {
        const long long row = t / gpr;
        const long long q = L.at((int)(t - row * gpr) * 4, (int)(row % L.ny), (int)(row / L.ny));
        Vec<float, 4> a = ldv<float, 4>(acc_a + q), b = ldv<float, 4>(acc_b + q);
        const Vec<float, 4> h = ldv<float, 4>(hi + q);
        const Vec<lo_code, 4> c = ldv<lo_code, 4>(lo + q);
#pragma unroll
        for (int e = 0; e < 4; ++e) accumulate_f32k(a.v[e], b.v[e], h.v[e], lo_decode(h.v[e], __ushort_as_half(c.v[e])));
        stv<float, 4>(acc_a + q, a);
        stv<float, 4>(acc_b + q, b);
    }
}

// out = scale * acc - shift (dense); with SUM the same pass leaves per-block partial sums of scale*acc
template <typename TO, bool F64, bool SUM, int W, typename I>
__global__ void __launch_bounds__(kThreads) k_grad(const void* acc_a, const void* acc_b, TO* __restrict__ out, Layout L,
                                                   double scale, double shift, double* partial) {
    double sum = 0.0;
    for_groups<W, I>(L, [&](const Group<I>& g) {
        const long long q = L.at(g.i0, g.j, g.k);
        Vec<TO, W> o;
#pragma unroll
        for (int e = 0; e < W; ++e) {
            double a;
            if constexpr (F64)
                a = ((const double*)acc_a)[q + e];
            else
                a = __dadd_rn(widen(((const float*)acc_a)[q + e]), widen(((const float*)acc_b)[q + e]));
            const double gval = __dmul_rn(scale, a);
            if constexpr (SUM) sum += gval;
            o.v[e] = (TO)(shift == 0.0 ? gval : __dsub_rn(gval, shift));
        }
        stv<TO, W>(out + g.dense, o);
    });
    if constexpr (SUM) {
        __shared__ double sh[32];
        const double v = block_sum(sum, sh);
        if (threadIdx.x == 0) partial[blockIdx.x] = v;
    }
}

__global__ void k_finish_sum(const double* partial, int n, double* out) {
    __shared__ double sh[32];
    double v = 0.0;
    for (int b = threadIdx.x; b < n; b += blockDim.x) v += partial[b];
    v = block_sum(v, sh);
    if (threadIdx.x == 0) *out = v;
}

// f(dtype tag, FP64 grid?) with compile-time values
template <class F>
void by_type(bool f64_data, bool f64_grid, F&& f) {
    if (f64_data)
        f64_grid ? f(0.0, std::true_type()) : f(0.0, std::false_type());
    else
        f64_grid ? f(0.f, std::true_type()) : f(0.f, std::false_type());
}

}  // namespace

int adjoint_inject(hg_grid* a, const void* v, int vdt) {
    hg_grid* g = a;
    by_type(vdt == HG_DT_F64, a->prec == HG_PREC_F64, [&](auto in, auto f64) {
        using T = decltype(in);
        dispatch_groups<T>(a->L, dense_width<T>(a->L, {v}), [&](auto W, auto I) {
            k_inject<T, f64.value, W.value, decltype(I)><<<group_blocks(a->L, W), kThreads, 0, a->stream>>>(
                (const T*)v, a->phi[a->cur], a->lo[a->cur], a->dlt[a->dcur], a->L);
        });
    });
    HG_LAUNCHED("adjoint injection kernel");
    return HG_OK;
}

int adjoint_accumulate(hg_grid* a, void* acc_a, void* acc_b) {
    hg_grid* g = a;
    const unsigned gpr = (unsigned)((a->nx + 3) / 4);
    const long long n = ((long long)gpr * a->ny * a->nz + kThreads - 1) / kThreads;
    const unsigned blocks = (unsigned)(n < (1LL << 22) ? n : 1LL << 22);
    k_accumulate<<<blocks, kThreads, 0, a->stream>>>((const float*)a->phi[a->cur], (const lo_code*)a->lo[a->cur],
                                                     (float*)acc_a, (float*)acc_b, a->L, gpr);
    HG_LAUNCHED("adjoint accumulation kernel");
    return HG_OK;
}

// dL/drho = -(c dt)^2 4 pi G * acc (dense, into out of type odt on the device), minus its mean when periodic
int adjoint_gradient(hg_grid* a, const void* acc_a, const void* acc_b, void* out, int odt, double* scratch) {
    hg_grid* g = a;
    const double scale = -a->src;
    auto pass = [&](auto sum, double shift) {
        by_type(odt == HG_DT_F64, a->prec == HG_PREC_F64, [&](auto o, auto f64) {
            using TO = decltype(o);
            dispatch_groups<TO>(a->L, dense_width<TO>(a->L, {out}), [&](auto W, auto I) {
                const unsigned blocks = sum.value ? (unsigned)kRedBlocks : group_blocks(a->L, W);
                k_grad<TO, f64.value, sum.value, W.value, decltype(I)>
                    <<<blocks, kThreads, 0, a->stream>>>(acc_a, acc_b, (TO*)out, a->L, scale, shift, scratch);
            });
        });
    };
    if (a->bc != HG_BC_PERIODIC) {
        pass(std::false_type(), 0.0);
        HG_LAUNCHED("adjoint gradient kernel");
        return HG_OK;
    }
    pass(std::true_type(), 0.0);
    HG_LAUNCHED("adjoint gradient kernel");
    k_finish_sum<<<1, kThreads, 0, a->stream>>>(scratch, kRedBlocks, scratch + kRedBlocks);
    HG_LAUNCHED("adjoint gradient sum kernel");
    double sum = 0.0;
    HG_CUDA(cudaMemcpyAsync(&sum, scratch + kRedBlocks, sizeof(double), cudaMemcpyDeviceToHost, a->stream));
    HG_CUDA(cudaStreamSynchronize(a->stream));
    const double mean = sum / ((double)a->nx * a->ny * a->nz);
    pass(std::false_type(), mean);
    HG_LAUNCHED("adjoint gradient kernel");
    return HG_OK;
}

}  // namespace hg
