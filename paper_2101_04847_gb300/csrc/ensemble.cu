// Ensembles of independent realisations (the paper runs at least 10 per
// experiment, Section 2): members may differ in grid size, physics and storage type;
// each is a full lbm_handle (init, diagnostics, fields, checkpoints) that only the
// ensemble steps.  The members of one storage type form chains; one launch per time
// step advances a chain (ensemble_step_kernel, step_kernels.cu: the single-grid tile
// code over a flat list of its members' tiles).  Members never wait for one another, so
// the chains run side by side on streams of their own, joined at the end of a call: one
// chain's blocks fill the SMs that the end of another's launch leaves idle.  Chunks of
// steps are captured in CUDA graphs.
#include "lbm_internal.cuh"

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

namespace {

constexpr int kEnsGraphChunk = 50;
constexpr int kEnsMaxMembers = 256;
constexpr int kTuneMinRows = 12;   // shortest tile that lbm_ens_tune tries itself

lbm_status ens_fail(lbm_status st, const std::string& msg) {
    lbm::set_last_error(msg);
    return st;
}

#define ENS_TRY(call, what)                                                                       \
    do {                                                                                          \
        cudaError_t e_ = (call);                                                                  \
        if (e_ != cudaSuccess) return ens_fail(LBM_ECUDA, std::string(what) + ": " + cudaGetErrorString(e_)); \
    } while (0)

}  // namespace

// Members of one storage type advanced by one launch per time step.
struct EnsChain {
    lbm::EnsKernel kernel;
    int storage = 0;
    std::vector<lbm_handle*> members;
    int begin = 0;        // its first member in the table
    int tiles = 0;
    cudaStream_t stream = nullptr;   // the ensemble's own for the first chain
    cudaEvent_t done = nullptr;      // the other chains': joins them to the ensemble's stream
};

struct lbm_ensemble {
    std::vector<lbm_handle*> members;
    std::vector<EnsChain> chains;
    std::vector<lbm::EnsMember> table;
    lbm::EnsMember* d_table = nullptr;
    int tile_x = lbm::kEnsAuto;      // 128 or 256 columns per tile (one per thread), or kEnsAuto
    int tile_y = 0;       // requested rows per tile; 0: chosen from the device's block slots
    int rows = 0;         // rows per tile in use
    int parity = 0;
    int64_t step = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    cudaEvent_t fork = nullptr;
    cudaGraphExec_t graph[2] = {nullptr, nullptr};
};

namespace {

void ens_drop_graphs(lbm_ensemble* e) {
    for (auto& g : e->graph) {
        if (g) cudaGraphExecDestroy(g);
        g = nullptr;
    }
}

int tiles_of(const lbm::Grid& g, int tile_x, int rows, int* tx, int* ty) {
    *tx = (g.nx + tile_x - 1) / tile_x;
    *ty = std::min(g.ny, std::max(1, (g.ny + rows - 1) / rows));
    return *tx * *ty;
}

// Rows per tile when none is requested: about two waves of tiles over all chains together.
// Short tiles read more halo rows, tall ones leave the chains too few blocks to fill the
// slots the others leave.  us per step: ten FP32 256x512 members 41.3 with 2 rows, 35.8
// with 4, 41.8 with 12 (0.9 waves); sixteen FP16 512x1024 120.9 with 16, 117.7 with 24, 132
// with 48; ten FP32 1024x2048 502 with 16, 485 with 48 and 64, 539 with 187 (one wave).  A
// launch that fits the slots is fastest with one row (one 128x256 member 4.0, 4.6 with 2);
// beyond that two rows are the least that pay (eight 128x256 members 14.5 with 1, 10.2).
constexpr int kMaxAutoRows = 48;
constexpr int kWideRows = 16;     // FP32 tiles of so many rows are 256 columns wide
int auto_rows(double waves_of_one_row) {
    if (waves_of_one_row <= 1.0) return 1;
    return std::max(2, (int)std::ceil(std::min(waves_of_one_row / 2.0, (double)kMaxAutoRows)));
}

// The chains of an ensemble: its members by storage type, each type's in up to
// kChainsPerType chains of about equal size.  Two cover each other's ends of launches
// (sixteen FP16 512x1024 members 140 us a step in one chain, 118 in two; ten FP32
// 1024x2048 511 and 485); more gain nothing further (116 to 121, 485).
constexpr int kChainsPerType = 2;
lbm_status ens_build_chains(lbm_ensemble* e) {
    for (int st : {LBM_STORE_F32, LBM_STORE_F16, LBM_STORE_BF16}) {
        std::vector<lbm_handle*> of;
        for (lbm_handle* h : e->members)
            if (lbm::handle_params(h).storage == st) of.push_back(h);
        const int n = std::min<int>(kChainsPerType, (int)of.size());
        std::vector<EnsChain> part(n);
        std::vector<double> size(n, 0.0);
        auto sites = [](lbm_handle* h) { return (double)lbm::handle_grid(h).nx * lbm::handle_grid(h).ny; };
        std::stable_sort(of.begin(), of.end(), [&](lbm_handle* a, lbm_handle* b) { return sites(a) > sites(b); });
        for (lbm_handle* h : of) {   // the largest first, each to the smallest chain
            const int k = (int)(std::min_element(size.begin(), size.end()) - size.begin());
            part[k].members.push_back(h);
            size[k] += sites(h);
        }
        for (EnsChain& c : part) {
            c.storage = st;
            if (e->chains.empty()) {
                c.stream = e->stream;
            } else {
                cudaError_t err = cudaStreamCreateWithFlags(&c.stream, cudaStreamNonBlocking);
                if (err == cudaSuccess) err = cudaEventCreateWithFlags(&c.done, cudaEventDisableTiming);
                if (err != cudaSuccess) {
                    if (c.stream) cudaStreamDestroy(c.stream);
                    return ens_fail(LBM_ECUDA, std::string("ensemble stream: ") + cudaGetErrorString(err));
                }
            }
            e->chains.push_back(c);
        }
    }
    if (e->chains.size() > 1)
        ENS_TRY(cudaEventCreateWithFlags(&e->fork, cudaEventDisableTiming), "ensemble event");
    return LBM_OK;
}

// (Re)build the member table for the current tile shape and upload it.
lbm_status ens_build_table(lbm_ensemble* e) {
    e->table.clear();
    double waves = 0.0;   // of one-row tiles, all chains
    for (EnsChain& c : e->chains) {
        c.kernel = lbm::ensemble_kernel(c.storage, e->tile_x);
        int slots = 1, tx, ty;
        ENS_TRY(lbm::ensemble_slots(c.kernel, &slots), "ensemble occupancy");
        for (lbm_handle* h : c.members) waves += (double)tiles_of(lbm::handle_grid(h), c.kernel.cols, 1, &tx, &ty) / slots;
    }
    e->rows = e->tile_y > 0 ? e->tile_y : auto_rows(waves);
    for (EnsChain& c : e->chains) {
        // tall FP32 tiles: 256 columns, as on one grid (ten 1024x2048 members 486 -> 461 us a
        // step, sixteen 512x1024 209 -> 192; short ones lose, eight 128x256 10 -> 13)
        if (e->tile_x == lbm::kEnsAuto && c.storage == LBM_STORE_F32 && e->rows >= kWideRows) {
            c.kernel = lbm::ensemble_kernel(c.storage, lbm::kWideTileW);
            int slots = 1;
            ENS_TRY(lbm::ensemble_slots(c.kernel, &slots), "ensemble occupancy");
        }
        c.begin = (int)e->table.size();
        c.tiles = 0;
        for (lbm_handle* h : c.members) {
            lbm::EnsMember m;
            m.grid = lbm::handle_grid(h);
            m.phys = lbm::handle_phys(h);
            m.buf[0] = lbm::handle_buffer(h, 0);
            m.buf[1] = lbm::handle_buffer(h, 1);
            m.flag = lbm::handle_flag(h);
            m.step_ctr = lbm::handle_step_counters(h);
            const int tiles = tiles_of(m.grid, c.kernel.cols, e->rows, &m.tiles_x, &m.tiles_y);
            m.tile_begin = c.tiles;
            c.tiles += tiles;
            e->table.push_back(m);
        }
    }
    ENS_TRY(cudaMemcpyAsync(e->d_table, e->table.data(), e->table.size() * sizeof(lbm::EnsMember),
                            cudaMemcpyHostToDevice, e->stream), "upload member table");
    ENS_TRY(cudaStreamSynchronize(e->stream), "sync");
    ens_drop_graphs(e);
    return LBM_OK;
}

// n steps from the given parity: the chains fork from the ensemble's stream and join it
// again whatever happens in between.
cudaError_t ens_launch_steps(lbm_ensemble* e, int parity, int64_t n) {
    cudaError_t err = cudaSuccess;
    if (n <= 0) return err;
    if (e->chains.size() > 1 && (err = cudaEventRecord(e->fork, e->stream)) != cudaSuccess) return err;
    for (EnsChain& c : e->chains) {
        const bool side = c.stream != e->stream;
        cudaError_t ce = side ? cudaStreamWaitEvent(c.stream, e->fork, 0) : cudaSuccess;
        for (int64_t k = 0; k < n && ce == cudaSuccess; ++k)
            ce = lbm::launch_ensemble_step(c.kernel, e->d_table + c.begin, (int)c.members.size(), c.tiles,
                                           (int)((parity + k) & 1), c.stream);
        if (err == cudaSuccess) err = ce;
    }
    for (EnsChain& c : e->chains)
        if (c.stream != e->stream) {
            cudaError_t ce = cudaEventRecord(c.done, c.stream);
            if (ce == cudaSuccess) ce = cudaStreamWaitEvent(e->stream, c.done, 0);
            if (err == cudaSuccess) err = ce;
        }
    return err;
}

lbm_status ens_launch(lbm_ensemble* e, int64_t n) {
    ENS_TRY(ens_launch_steps(e, e->parity, n), "ensemble step");
    e->parity ^= (int)(n & 1);
    return LBM_OK;
}

// n steps from the given parity as a graph.
lbm_status ens_capture(lbm_ensemble* e, int parity, int n, cudaGraphExec_t* out) {
    cudaGraph_t g = nullptr;
    ENS_TRY(cudaStreamBeginCapture(e->stream, cudaStreamCaptureModeThreadLocal), "begin capture");
    cudaError_t err = ens_launch_steps(e, parity, n);
    const cudaError_t end = cudaStreamEndCapture(e->stream, &g);
    if (err == cudaSuccess) err = end;
    if (err != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return ens_fail(LBM_ECUDA, std::string("capture ensemble step: ") + cudaGetErrorString(err));
    }
    err = cudaGraphInstantiate(out, g, 0);
    cudaGraphDestroy(g);
    if (err != cudaSuccess) return ens_fail(LBM_ECUDA, std::string("instantiate: ") + cudaGetErrorString(err));
    return LBM_OK;
}

lbm_status ens_graph(lbm_ensemble* e, cudaGraphExec_t* out) {
    const int par = e->parity;
    if (!e->graph[par]) {
        const lbm_status st = ens_capture(e, par, kEnsGraphChunk, &e->graph[par]);
        if (st != LBM_OK) return st;
    }
    *out = e->graph[par];
    return LBM_OK;
}

// ms per step with the tile shape in use, by events a and b around replays of a graph of
// kTuneSteps steps (single launches would time the host where a step takes a few us); more
// replays where they are short, 32 steps in all at most.  The parity, an even number of
// steps on, is the same; the members' states have to be restored.
constexpr int kTuneSteps = 4;
lbm_status ens_time(lbm_ensemble* e, cudaEvent_t a, cudaEvent_t b, double* ms_per_step) {
    cudaGraphExec_t g = nullptr;
    const lbm_status st = ens_capture(e, e->parity, kTuneSteps, &g);
    if (st != LBM_OK) return st;
    cudaError_t err = cudaGraphLaunch(g, e->stream);
    float ms = 0.0f;
    for (int replays : {1, 6}) {
        if (err == cudaSuccess) err = cudaEventRecord(a, e->stream);
        for (int k = 0; k < replays && err == cudaSuccess; ++k) err = cudaGraphLaunch(g, e->stream);
        if (err == cudaSuccess) err = cudaEventRecord(b, e->stream);
        if (err == cudaSuccess) err = cudaEventSynchronize(b);
        if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, a, b);
        if (err != cudaSuccess) break;
        *ms_per_step = ms / (replays * kTuneSteps);
        if (ms > 0.2f) break;
    }
    cudaGraphExecDestroy(g);
    if (err != cudaSuccess) return ens_fail(LBM_ECUDA, std::string("timing: ") + cudaGetErrorString(err));
    return LBM_OK;
}

}  // namespace

extern "C" {

void lbm_ens_destroy(lbm_ensemble* e) {
    if (!e) return;
    if (e->stream) cudaStreamSynchronize(e->stream);
    ens_drop_graphs(e);
    for (lbm_handle* h : e->members) {
        lbm::handle_set_ensemble(h, false);
        lbm_destroy(h);
    }
    for (EnsChain& c : e->chains) {
        if (c.done) cudaEventDestroy(c.done);
        if (c.stream && c.stream != e->stream) cudaStreamDestroy(c.stream);
    }
    if (e->fork) cudaEventDestroy(e->fork);
    if (e->d_table) cudaFree(e->d_table);
    if (e->own_stream && e->stream) cudaStreamDestroy(e->stream);
    delete e;
}

lbm_status lbm_ens_create(int32_t n, const lbm_params* params, void* cuda_stream, lbm_ensemble** out) {
    if (!out) return ens_fail(LBM_EINVAL, "out is NULL");
    *out = nullptr;
    if (!params || n < 1 || n > kEnsMaxMembers) return ens_fail(LBM_EINVAL, "need 1..256 member parameter sets");
    lbm_ensemble* e = new lbm_ensemble();
    if (cuda_stream) {
        e->stream = (cudaStream_t)cuda_stream;
    } else {
        cudaError_t err = cudaStreamCreateWithFlags(&e->stream, cudaStreamNonBlocking);
        if (err != cudaSuccess) {
            delete e;
            return ens_fail(LBM_ECUDA, std::string("create stream: ") + cudaGetErrorString(err));
        }
        e->own_stream = true;
    }
    e->tile_y = params[0].tile_y > 0 ? params[0].tile_y : 0;
    e->tile_x = params[0].tile_x == lbm::kWideTileW || params[0].tile_x == lbm::kBlockTileW ? params[0].tile_x
                                                                                             : lbm::kEnsAuto;
    for (int i = 0; i < n; ++i) {
        lbm_params p = params[i];
        p.kernel = LBM_KERNEL_STAGED;
        lbm_handle* h = nullptr;
        lbm_status st = lbm_create_ex(&p, nullptr, 0, e->stream, &h);
        if (st != LBM_OK) {
            const std::string msg = std::string("member ") + std::to_string(i) + ": " + lbm_last_error();
            lbm_ens_destroy(e);
            return ens_fail(st, msg);
        }
        lbm::handle_set_ensemble(h, true);
        e->members.push_back(h);
    }
    cudaError_t err = cudaMalloc((void**)&e->d_table, (size_t)n * sizeof(lbm::EnsMember));
    if (err != cudaSuccess) {
        e->d_table = nullptr;
        lbm_ens_destroy(e);
        return ens_fail(LBM_ENOMEM, "member table");
    }
    lbm_status st = ens_build_chains(e);
    if (st == LBM_OK) st = ens_build_table(e);
    if (st != LBM_OK) {
        const std::string msg = lbm_last_error();
        lbm_ens_destroy(e);
        return ens_fail(st, msg);
    }
    *out = e;
    return LBM_OK;
}

lbm_status lbm_ens_step(lbm_ensemble* e, int64_t nsteps) {
    if (!e) return ens_fail(LBM_EINVAL, "ensemble is NULL");
    if (nsteps < 0) return ens_fail(LBM_EINVAL, "nsteps must be >= 0");
    int64_t left = nsteps;
    while (left >= kEnsGraphChunk) {
        cudaGraphExec_t g = nullptr;
        lbm_status st = ens_graph(e, &g);
        if (st != LBM_OK) return st;
        ENS_TRY(cudaGraphLaunch(g, e->stream), "graph launch");
        e->parity ^= (kEnsGraphChunk & 1);
        left -= kEnsGraphChunk;
    }
    lbm_status st = ens_launch(e, left);
    if (st != LBM_OK) return st;
    e->step += nsteps;
    for (lbm_handle* h : e->members) lbm::handle_advance(h, nsteps);
    return LBM_OK;
}

lbm_status lbm_ens_sync(lbm_ensemble* e) {
    if (!e) return ens_fail(LBM_EINVAL, "ensemble is NULL");
    lbm_status worst = LBM_OK;
    for (lbm_handle* h : e->members) {
        lbm_status st = lbm::handle_check(h);
        if (st != LBM_OK && worst == LBM_OK) worst = st;
    }
    return worst;
}

lbm_status lbm_ens_member(lbm_ensemble* e, int32_t i, lbm_handle** out) {
    if (!e || !out) return ens_fail(LBM_EINVAL, "NULL argument");
    if (i < 0 || i >= (int)e->members.size()) return ens_fail(LBM_EINVAL, "member index out of range");
    *out = e->members[i];
    return LBM_OK;
}

lbm_status lbm_ens_diagnostics(lbm_ensemble* e, lbm_diag* out) {
    if (!e || !out) return ens_fail(LBM_EINVAL, "NULL argument");
    lbm_status worst = LBM_OK;
    for (size_t i = 0; i < e->members.size(); ++i) {
        lbm_status st = lbm_diagnostics(e->members[i], &out[i]);
        if (st != LBM_OK && worst == LBM_OK) worst = st;
    }
    return worst;
}

lbm_status lbm_ens_tune(lbm_ensemble* e, int32_t* tile_y_out, double* ms_out) {
    if (!e) return ens_fail(LBM_EINVAL, "ensemble is NULL");
    const int cand[] = {0, 12, 16, 20, 24, 32, 48, 64, 96};   // 0: the default where it is no shorter
    const int widths[] = {lbm::kEnsAuto, lbm::kBlockTileW, lbm::kWideTileW};
    static_assert(kTuneMinRows == 12, "the shortest candidate");
    cudaEvent_t a, b;
    ENS_TRY(cudaEventCreate(&a), "event");
    ENS_TRY(cudaEventCreate(&b), "event");
    // the shape found: it stays where no candidate is faster, and after an error (eight
    // 128x256 members keep their 2 rows and 9.9 us a step; 15.9 with 12 rows)
    const int found_tx = e->tile_x, found_ty = e->tile_y;
    auto shape = [&](int tx, int ty) {
        e->tile_x = tx;
        e->tile_y = ty;
        return ens_build_table(e);
    };
    auto timed = [&](double* ms) {
        const lbm_status st = ens_time(e, a, b, ms);
        for (lbm_handle* h : e->members) ENS_TRY(lbm::handle_restore_state(h), "restore state");
        return st;
    };
    auto tune = [&]() -> lbm_status {
        for (lbm_handle* h : e->members) ENS_TRY(lbm::handle_save_state(h), "save state");
        double found_ms = 0.0, best_ms = 1e30;
        lbm_status st = timed(&found_ms);
        if (st != LBM_OK) return st;
        int best_tx = found_tx, best_ty = found_ty, best_rows = 0;
        for (int tx : widths)
            for (int ty : cand) {
                if ((st = shape(tx, ty)) != LBM_OK) return st;
                if (e->rows < kTuneMinRows) continue;
                double ms = 0.0;
                if ((st = timed(&ms)) != LBM_OK) return st;
                if (ms < best_ms) {
                    best_ms = ms;
                    best_tx = tx;
                    best_ty = ty;
                    best_rows = e->rows;
                }
            }
        // the least of many noisy timings is below what it stands for: both once more
        double again_ms = 0.0;
        if ((st = shape(found_tx, found_ty)) != LBM_OK || (st = timed(&again_ms)) != LBM_OK) return st;
        found_ms = std::min(found_ms, again_ms);
        if ((st = shape(best_tx, best_ty)) != LBM_OK || (st = timed(&best_ms)) != LBM_OK) return st;
        const bool faster = best_ms < found_ms;
        if (!faster && (st = shape(found_tx, found_ty)) != LBM_OK) return st;
        if (tile_y_out) *tile_y_out = e->rows >= kTuneMinRows ? e->rows : best_rows;
        if (ms_out) *ms_out = faster ? best_ms : found_ms;
        return LBM_OK;
    };
    lbm_status st = tune();
    if (st != LBM_OK) {
        const std::string msg = lbm_last_error();
        shape(found_tx, found_ty);
        lbm::set_last_error(msg);
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    return st;
}

lbm_status lbm_ens_tile_width(lbm_ensemble* e, int32_t* tile_x) {
    if (!e || !tile_x) return ens_fail(LBM_EINVAL, "NULL argument");
    *tile_x = e->tile_x;
    return LBM_OK;
}

}  // extern "C"
