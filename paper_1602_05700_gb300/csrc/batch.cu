// Many independent grids advanced together (the batching workload: uneven sizes, mixed precisions).
//
// One sub-step of every grid is one batched launch of the flat sweep (stencil.cu, k_batch_flat: block -> grid by a prefix
// table; FP64 and float blocks alternate, so that FP64- and integer-bound and HBM-bound ones share the SMs; boundary ghosts
// are written inside the launch); float grids large enough for the TMA-staged sweep are a second launch beside it.
// hg_batch_step(b, n) records the n sub-steps once as a CUDA graph on the batch's own stream and replays it with a
// single graph launch; the kernels read the per-grid arguments from two device tables (for the two time-level
// parities), refreshed from the grids before every replay, so the graph stays valid while the grids' states move on.
// Results are identical to stepping each grid on its own: the per-cell arithmetic is the same code.
//
// 48 grids of 64^3 to 192^3, alternating precisions, per sub-step: 2.18 ms with marching FP64 blocks and TMA-staged float
// blocks in one launch (the FP64 half latency-bound at 16 warps per SM, 60% of a 96-cell row's tile in use), 1.05 with
// the flat sweep (sweep_flat.cuh says what it changes).
//
// Autotuning: two knobs of the launch are chosen by timing the first sub-steps of the first hg_batch_step with CUDA
// events -- every candidate computes the same result, so the timing runs are real sub-steps -- and cached per
// (device, set of grid shapes/precisions/boundaries) for the process:
//   * one flat launch per sub-step for both precisions, or two (split mode: an FP64 launch and a float launch per
//     sub-step, as two independent chains on two streams);
//   * the z extent of a TMA-staged block of the large float grids (8 or 16 planes).
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "hg_internal.cuh"

using namespace hg;

struct hg_batch {
    int n;
    std::vector<hg_grid*> grids;
    int device;
    cudaStream_t stream;  // own non-blocking stream (graphs cannot be captured on the legacy default stream)
    cudaEvent_t ev_in, ev_out;
    BatchEntry* d_tab[2];  // per-grid entries, per parity: FP64 grids, then float ones, then large float ones
    unsigned* d_first;     // the three classes' prefix tables of block numbers, each with one entry more than grids
    int n64, n32, nbig;
    unsigned blocks64, blocks32, blocksbig;
    int zb;    // 0 until tuned, then 1: planes of a flat block
    int zb32;  // z planes per block of the large float grids (TMA-staged)
    int split; // 1: FP64 and float entries as two launches per sub-step, on two streams
    int force_split;  // -1: the autotuner chooses split; 0 or 1: pinned by hg_batch_set_split
    cudaStream_t stream2;
    cudaEvent_t ev_fork, ev_join;
    // graph of `graph_steps` sub-steps
    cudaGraph_t graph;
    cudaGraphExec_t exec;
    int graph_steps;
};

namespace {

std::mutex g_tune_mu;
struct Tuning {
    int zb32, split;
};
std::map<std::string, Tuning> g_tuned;  // autotuner cache: key -> the chosen launch

std::string tune_key(const hg_batch* b) {
    cudaDeviceProp p;
    cudaGetDeviceProperties(&p, b->device);
    std::vector<std::string> parts;
    for (hg_grid* g : b->grids) {
        char buf[96];
        snprintf(buf, sizeof buf, "%dx%dx%d/%d/%d", g->nx, g->ny, g->nz, g->prec, g->bc);
        parts.push_back(buf);
    }
    std::sort(parts.begin(), parts.end());
    std::string k = p.name;
    for (auto& s : parts) k += ";" + s;
    k += ";split=" + std::to_string(b->force_split);
    return k;
}

// FP64 grids, float grids of the flat sweep, large float grids; largest first within a class
int class_of(const hg_grid* g) { return g->prec == HG_PREC_F64 ? 0 : flat_sized(g) ? 1 : 2; }
std::vector<hg_grid*> launch_order(const hg_batch* b) {
    std::vector<hg_grid*> o(b->grids);
    auto cells = [](const hg_grid* g) { return (long long)g->nx * g->ny * g->nz; };
    std::stable_sort(o.begin(), o.end(), [&](const hg_grid* a, const hg_grid* c) {
        if (class_of(a) != class_of(c)) return class_of(a) < class_of(c);
        return cells(a) > cells(c);
    });
    return o;
}

// device tables for the sub-steps that start from parity p (0: every grid's current level, 1: the next one)
int upload_tables(hg_batch* b) {
    std::vector<BatchEntry> tab[2];
    const std::vector<hg_grid*> order = launch_order(b);
    for (int p = 0; p < 2; ++p) {
        for (hg_grid* g : order) {
            const int cur = g->cur;
            g->cur = cur ^ p;
            BatchEntry e;
            memset(&e, 0, sizeof e);
            int rc = HG_OK;
            if (class_of(g) == 2) {
                rc = tma_entry(g, &e, b->zb32);
            } else {
                e.A = sweep_args(g, 0);
                e.G = flat_grid(g, kBatchThreads, g->prec == HG_PREC_F32K ? 4 : 1);
                e.err = g->derr;
            }
            g->cur = cur;
            if (rc) return rc;
            tab[p].push_back(e);
        }
    }
    int n[3] = {0, 0, 0};
    unsigned blocks[3];
    std::vector<unsigned> first;
    for (hg_grid* g : order) ++n[class_of(g)];
    for (int c = 0, i = 0; c < 3; ++c) {
        first.push_back(0);
        for (int e = 0; e < n[c]; ++e, ++i)
            first.push_back(first.back() + (c == 2 ? sweep_blocks(tab[0][i].A)
                                                   : (tab[0][i].G.tiles + kBatchTiles - 1) / kBatchTiles));
        blocks[c] = first.back();
    }
    b->n64 = n[0], b->n32 = n[1], b->nbig = n[2];
    b->blocks64 = blocks[0], b->blocks32 = blocks[1], b->blocksbig = blocks[2];
    for (int p = 0; p < 2; ++p)
        HG_CUDA(cudaMemcpyAsync(b->d_tab[p], tab[p].data(), tab[p].size() * sizeof(BatchEntry), cudaMemcpyHostToDevice,
                                b->stream));
    HG_CUDA(cudaMemcpyAsync(b->d_first, first.data(), first.size() * sizeof(unsigned), cudaMemcpyHostToDevice, b->stream));
    HG_CUDA(cudaStreamSynchronize(b->stream));  // the host vectors go out of scope
    return HG_OK;
}

// The launches of `count` sub-steps, the first of parity p0.  The second stream, forked from and joined back into the
// batch stream, carries the large float grids and in split mode every float grid (the chains touch different grids, so
// they need no ordering between them).
int enqueue_substeps(hg_batch* b, int p0, int count) {
    int rc = HG_OK;
    const bool second = b->nbig > 0 || (b->split && b->n32 > 0);
    if (second) {
        HG_CUDA(cudaEventRecord(b->ev_fork, b->stream));
        HG_CUDA(cudaStreamWaitEvent(b->stream2, b->ev_fork, 0));
    }
    const unsigned *f64 = b->d_first, *f32 = f64 + b->n64 + 1, *fbig = f32 + b->n32 + 1;
    for (int s = 0; s < count && rc == HG_OK; ++s) {
        const BatchEntry *t64 = b->d_tab[(p0 + s) & 1], *t32 = t64 + b->n64, *tbig = t32 + b->n32;
        if (b->split) {
            rc = launch_batch_flat(b->stream, t64, f64, b->n64, b->blocks64, t32, f32, 0, 0u);
            if (rc == HG_OK) rc = launch_batch_flat(b->stream2, t64, f64, 0, 0u, t32, f32, b->n32, b->blocks32);
        } else {
            rc = launch_batch_flat(b->stream, t64, f64, b->n64, b->blocks64, t32, f32, b->n32, b->blocks32);
        }
        if (rc == HG_OK) rc = launch_batch_tma(b->stream2, tbig, fbig, b->nbig, b->blocksbig);
    }
    if (!second) return rc;
    // join even after an error, so that a capture in progress ends with both streams in it
    cudaError_t e1 = cudaEventRecord(b->ev_join, b->stream2);
    cudaError_t e2 = cudaStreamWaitEvent(b->stream, b->ev_join, 0);
    if (rc) return rc;
    if (e1 != cudaSuccess) return cuda_fail(e1, "cudaEventRecord");
    if (e2 != cudaSuccess) return cuda_fail(e2, "cudaStreamWaitEvent");
    return HG_OK;
}

void advance(hg_batch* b, int n) {
    for (hg_grid* g : b->grids) {
        if (n & 1) g->cur ^= 1;
        g->step += n;
    }
}

// pick the launch by timing two sub-steps per candidate (real sub-steps: every candidate gives the same result);
// returns the number of sub-steps taken in *taken
int autotune(hg_batch* b, int budget, int* taken) {
    *taken = 0;
    const std::string key = tune_key(b);
    {
        std::lock_guard<std::mutex> lock(g_tune_mu);
        auto it = g_tuned.find(key);
        if (it != g_tuned.end()) {
            b->zb = 1;
            b->zb32 = it->second.zb32;
            b->split = it->second.split;
            return upload_tables(b);
        }
    }
    bool any64 = false, any32 = false, anybig = false;
    for (hg_grid* g : b->grids) {
        any64 = any64 || class_of(g) == 0;
        any32 = any32 || class_of(g) == 1;
        anybig = anybig || class_of(g) == 2;
    }
    std::vector<Tuning> cand;
    cand.push_back({8, b->force_split > 0 ? 1 : 0});
    if (b->force_split < 0 && any64 && any32) cand.push_back({8, 1});
    Tuning best = cand[0];
    float best_ms = -1.f;
    cudaEvent_t e0, e1;
    HG_CUDA(cudaEventCreate(&e0));
    HG_CUDA(cudaEventCreate(&e1));
    int rc = HG_OK;
    bool complete = true;
    auto time_one = [&](const Tuning& t) -> bool {  // false: no budget left or an error (rc)
        if (*taken + 2 > budget) {
            complete = false;
            return false;
        }
        b->zb32 = t.zb32;
        b->split = t.split;
        if ((rc = upload_tables(b))) return false;
        cudaEventRecord(e0, b->stream);
        if ((rc = enqueue_substeps(b, 0, 2))) return false;  // two sub-steps (both parities) per candidate
        cudaEventRecord(e1, b->stream);
        cudaError_t e = cudaEventSynchronize(e1);
        if (e != cudaSuccess) {
            rc = cuda_fail(e, "autotuner timing");
            return false;
        }
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        advance(b, 2);
        *taken += 2;
        if (best_ms < 0.f || ms < best_ms) {
            best = t;
            best_ms = ms;
        }
        return true;
    };
    for (const Tuning& t : cand)
        if (!time_one(t)) break;
    if (rc == HG_OK && complete && anybig && best_ms >= 0.f) {
        Tuning t = best;
        t.zb32 = 16;
        time_one(t);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc) return rc;
    b->zb = 1;
    b->zb32 = best.zb32;  // too few sub-steps to time anything: the first candidate
    b->split = best.split;
    if (complete) {
        std::lock_guard<std::mutex> lock(g_tune_mu);
        g_tuned[key] = best;
    }
    return upload_tables(b);
}

void destroy_graph(hg_batch* b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    b->exec = nullptr;
    b->graph = nullptr;
    b->graph_steps = 0;
}

void release(hg_batch* b) {
    destroy_graph(b);
    void* ptrs[] = {b->d_tab[0], b->d_tab[1], b->d_first};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    cudaEvent_t evs[] = {b->ev_in, b->ev_out, b->ev_fork, b->ev_join};
    for (cudaEvent_t ev : evs)
        if (ev) cudaEventDestroy(ev);
    if (b->stream) cudaStreamDestroy(b->stream);
    if (b->stream2) cudaStreamDestroy(b->stream2);
}

}  // namespace

extern "C" {

int hg_batch_create(hg_grid* const* grids, int n, hg_batch** out) {
    HG_RANGE("hg_batch_create");
    if (!out) return fail(HG_ERR_ARG, "null output pointer");
    *out = nullptr;
    if (!grids || n < 1) return fail(HG_ERR_ARG, "need at least one grid");
    for (int i = 0; i < n; ++i) {
        if (!grids[i]) return fail(HG_ERR_ARG, "grid %d is null", i);
        if (grids[i]->device != grids[0]->device) return fail(HG_ERR_ARG, "all grids of a batch must share one device");
        if (grids[i]->ziface) return fail(HG_ERR_ARG, "grid %d is a slab (z interfaces): batches hold whole grids", i);
        if (grids[i]->stream != grids[0]->stream) return fail(HG_ERR_ARG, "all grids of a batch must share one stream");
        for (int j = 0; j < i; ++j)
            if (grids[j] == grids[i]) return fail(HG_ERR_ARG, "grid %d appears twice", i);
    }
    cudaError_t e = cudaSetDevice(grids[0]->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaSetDevice");
    hg_batch* b = new hg_batch();
    b->n = n;
    b->force_split = -1;
    b->grids.assign(grids, grids + n);
    b->device = grids[0]->device;
    int rc = HG_OK;
    auto ck = [&](cudaError_t err, const char* what) {
        if (rc == HG_OK && err != cudaSuccess) rc = cuda_fail(err, what);
    };
    ck(cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking), "cudaStreamCreate");
    ck(cudaStreamCreateWithFlags(&b->stream2, cudaStreamNonBlocking), "cudaStreamCreate");
    for (cudaEvent_t* ev : {&b->ev_in, &b->ev_out, &b->ev_fork, &b->ev_join})
        ck(cudaEventCreateWithFlags(ev, cudaEventDisableTiming), "cudaEventCreate");
    for (int p = 0; p < 2 && rc == HG_OK; ++p) ck(cudaMalloc(&b->d_tab[p], n * sizeof(BatchEntry)), "cudaMalloc(table)");
    ck(cudaMalloc(&b->d_first, (n + 3) * sizeof(unsigned)), "cudaMalloc(table)");
    if (rc == HG_OK) rc = upload_tables(b);
    if (rc != HG_OK) {
        release(b);
        delete b;
        return rc;
    }
    *out = b;
    return HG_OK;
}

int hg_batch_step(hg_batch* b, int n_substeps) {
    HG_RANGE("hg_batch_step");
    if (!b) return fail(HG_ERR_ARG, "null batch");
    if (n_substeps < 0) return fail(HG_ERR_ARG, "n_substeps must be >= 0");
    if (n_substeps == 0) return HG_OK;
    cudaError_t e = cudaSetDevice(b->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaSetDevice");
    cudaStream_t gs = b->grids[0]->stream;
    // the batch stream waits for earlier work of the grids, and the grids' stream for the batch
    HG_CUDA(cudaEventRecord(b->ev_in, gs));
    HG_CUDA(cudaStreamWaitEvent(b->stream, b->ev_in, 0));
    int rc = HG_OK;
    int done = 0;
    if (b->zb == 0) {
        rc = autotune(b, n_substeps, &done);
        if (rc) return rc;
        destroy_graph(b);
    }
    const int n = n_substeps - done;
    if (n > 0) {
        if ((rc = upload_tables(b))) return rc;
        if (b->graph_steps != n) {
            destroy_graph(b);
            HG_CUDA(cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal));
            rc = enqueue_substeps(b, 0, n);
            cudaGraph_t graph = nullptr;
            e = cudaStreamEndCapture(b->stream, &graph);
            if (rc) {
                if (graph) cudaGraphDestroy(graph);
                return rc;
            }
            if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
            b->graph = graph;
            HG_CUDA(cudaGraphInstantiate(&b->exec, b->graph, 0));
            b->graph_steps = n;
        }
        HG_CUDA(cudaGraphLaunch(b->exec, b->stream));
        advance(b, n);
    }
    HG_CUDA(cudaEventRecord(b->ev_out, b->stream));
    HG_CUDA(cudaStreamWaitEvent(gs, b->ev_out, 0));
    return HG_OK;
}

int hg_batch_set_split(hg_batch* b, int mode) {
    HG_RANGE("hg_batch_set_split");
    if (!b) return fail(HG_ERR_ARG, "null batch");
    if (mode < -1 || mode > 1) return fail(HG_ERR_ARG, "mode must be -1 (autotuned), 0 or 1");
    if (mode == b->force_split) return HG_OK;
    b->force_split = mode;
    b->zb = 0;  // the next hg_batch_step tunes (or finds in the cache) the launch for this mode
    destroy_graph(b);
    return HG_OK;
}

int hg_batch_info(const hg_batch* b, int* z_planes_per_block, long long* blocks_per_substep) {
    HG_RANGE("hg_batch_info");
    if (!b) return fail(HG_ERR_ARG, "null batch");
    if (z_planes_per_block) *z_planes_per_block = b->zb;
    if (blocks_per_substep) *blocks_per_substep = (long long)b->blocks64 + b->blocks32 + b->blocksbig;
    return HG_OK;
}

int hg_batch_tuning(const hg_batch* b, int out[4]) {
    HG_RANGE("hg_batch_tuning");
    if (!b || !out) return fail(HG_ERR_ARG, "null argument");
    out[0] = b->zb;
    out[1] = 0;
    out[2] = b->zb32;
    out[3] = b->split;
    return HG_OK;
}

void hg_batch_free(hg_batch* b) {
    HG_RANGE("hg_batch_free");
    if (!b) return;
    cudaSetDevice(b->device);
    cudaStreamSynchronize(b->stream);
    release(b);
    delete b;
}

}  // extern "C"
