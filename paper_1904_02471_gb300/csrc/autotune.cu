// Autotuner: picks the tile shape and grid size of every group by
// timing each candidate on the group's own lattices (state saved and
// restored around the trials). Results are cached for the life of the process
// per model, set, precision, scheme, recording interval and the lattices' sizes
// and storage: the tile and the kind of grid (GridKind), whose size follows the
// group.
#include <algorithm>
#include <cstdio>
#include <map>
#include <mutex>
#include <tuple>

#include "engine.h"

namespace lbm {

namespace {
// One block set per SM, two, one block per work item; none exceeds the items.
enum GridKind { GRID_PERSISTENT = 0, GRID_TWICE, GRID_ITEMS, GRID_KINDS };
int grid_of(int kind, int items, int persistent) {
    const int p = std::min(items, persistent);
    return std::max(1, kind == GRID_PERSISTENT ? p : (kind == GRID_TWICE ? std::min(items, 2 * p) : items));
}
using Key = std::tuple<int, int, int, int, long long, size_t, uint64_t>;
constexpr size_t CACHE_MAX = 4096;   // entries
std::map<Key, std::pair<int, int>>& cache() {   // tile, GridKind
    static std::map<Key, std::pair<int, int>> m;
    return m;
}
std::mutex& cache_mutex() {
    static std::mutex m;
    return m;
}
// 64-bit FNV-1a over the lattices' sizes and storage.
uint64_t add_hash(uint64_t h, uint64_t v) {
    for (int i = 0; i < 8; ++i) h = (h ^ ((v >> (8 * i)) & 255)) * 1099511628211ull;
    return h;
}
}  // namespace

int Engine::tune(int trial_steps, std::string* report) {
    if (trial_steps < 1) trial_steps = 1;
    std::string rep;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return cuda_fail(cudaGetLastError(), "cudaEventCreate");
    for (int gi = 0; gi < (int)groups.size(); ++gi) {
        Group& g = groups[gi];
        if (g.members.empty()) continue;
        uint64_t shapes = 14695981039346656037ull;
        for (int li : g.members) {
            shapes = add_hash(shapes, (uint64_t)lat[li].spec.nx << 32 | (uint32_t)lat[li].spec.ny);
            shapes = add_hash(shapes, (uint64_t)lat[li].spec.storage);
        }
        const Key key{g.model, g.q1, g.precision, g.scheme, g.min_every, g.members.size(), shapes};
        {
            std::lock_guard<std::mutex> lk(cache_mutex());
            auto it = cache().find(key);
            if (it != cache().end()) {
                int rc = apply_config(gi, it->second.first, 0);
                if (rc) return rc;
                g.grid = grid_of(it->second.second, g.total_items, persistent_grid(g, g.tile));
                char b[160];
                snprintf(b, sizeof b, "[g%d %s q%d %s cached tile=%d grid=%d] ", gi, g.model == LBM_CS ? "CS" : "FD", g.q1,
                         g.precision == LBM_FP64 ? "fp64" : "fp32", g.tile, g.grid);
                rep += b;
                continue;
            }
        }
        // save the state of the group's lattices
        std::vector<void*> saved;
        for (int li : g.members) {
            void* p = nullptr;
            cudaError_t e = cudaMalloc(&p, lat[li].state_bytes());
            if (e != cudaSuccess) {
                for (void* q : saved) cudaFree(q);
                return cuda_fail(e, "cudaMalloc(tune save)");
            }
            e = cudaMemcpyAsync(p, lat[li].mem, lat[li].state_bytes(), cudaMemcpyDeviceToDevice, stream_);
            if (e != cudaSuccess) return cuda_fail(e, "tune save copy");
            saved.push_back(p);
        }
        const int ntiles = g.model == LBM_CS ? (int)CS_NTILES : (int)FD_NALL;
        float best = 1e30f;
        int best_tile = g.tile, best_kind = GRID_PERSISTENT;
        // Trials record as the steps do (into slots that the steps write
        // again), except intervals longer than a trial, whose record would
        // weigh too much in it.
        std::vector<std::pair<int, long long>> every;
        for (int li : g.members)
            if (lat[li].obs_every > trial_steps) {
                every.emplace_back(li, lat[li].obs_every);
                lat[li].obs_every = 0;
            }
        struct Restore {
            std::vector<Lattice>& lat;
            std::vector<std::pair<int, long long>>& every;
            ~Restore() { now(); }
            void now() {
                for (const auto& e : every) lat[e.first].obs_every = e.second;
                every.clear();
            }
        } restore{lat, every};
        for (int t = 0; t < ntiles; ++t) {
            if (g.model == LBM_FD && !fd_variant_fits(g.precision, g.q1, t, g.scheme)) continue;
            int rc = apply_config(gi, t, 0);
            if (rc) return rc;
            const int pers = persistent_grid(g, t);
            for (int kind = 0; kind < GRID_KINDS; ++kind) {
                const int grid = grid_of(kind, g.total_items, pers);
                if (kind > 0 && grid == grid_of(kind - 1, g.total_items, pers)) continue;
                g.grid = grid;
                const GroupDev gd = g.dev();
                auto run = [&](int steps) -> cudaError_t {
                    for (int j = 0; j < steps; ++j) {
                        const int launches = g.model == LBM_CS ? 1 : fd_stages(g.scheme);
                        for (int st = 1; st <= launches; ++st) {
                            cudaError_t e = g.model == LBM_CS
                                                ? launch_cs_step(g.precision, g.tile, g.grid, gd, j, stream_)
                                                : launch_fd_stage(g.precision, g.q1, g.scheme, g.tile, g.grid, gd, j, st, stream_);
                            if (e == cudaSuccess && st == 1 && obs_launch(g))
                                e = launch_obs_finish(gd, (int)g.members.size(), g.total_items, g.grid, j, stream_);
                            if (e != cudaSuccess) return e;
                        }
                    }
                    return cudaSuccess;
                };
                cudaError_t e = run(1);
                if (e == cudaSuccess) e = cudaEventRecord(e0, stream_);
                if (e == cudaSuccess) e = run(trial_steps);
                if (e == cudaSuccess) e = cudaEventRecord(e1, stream_);
                if (e == cudaSuccess) e = cudaEventSynchronize(e1);
                if (e != cudaSuccess) return cuda_fail(e, "tune trial");
                float ms = 0;
                cudaEventElapsedTime(&ms, e0, e1);
                if (ms < best) {
                    best = ms;
                    best_tile = t;
                    best_kind = kind;
                }
            }
        }
        // restore state and apply the winner
        for (size_t m = 0; m < g.members.size(); ++m) {
            const Lattice& L = lat[g.members[m]];
            cudaError_t e = cudaMemcpyAsync(L.mem, saved[m], L.state_bytes(), cudaMemcpyDeviceToDevice, stream_);
            if (e != cudaSuccess) return cuda_fail(e, "tune restore copy");
        }
        cudaStreamSynchronize(stream_);
        for (void* p : saved) cudaFree(p);
        restore.now();
        int rc = apply_config(gi, best_tile, 0);
        if (rc) return rc;
        g.grid = grid_of(best_kind, g.total_items, persistent_grid(g, best_tile));
        {
            std::lock_guard<std::mutex> lk(cache_mutex());
            if (cache().size() >= CACHE_MAX) cache().clear();
            cache()[key] = {best_tile, best_kind};
        }
        char b[200];
        snprintf(b, sizeof b, "[g%d %s q%d %s tile=%dx%d grid=%d %.4f ms/step] ", gi, g.model == LBM_CS ? "CS" : "FD",
                 g.q1, g.precision == LBM_FP64 ? "fp64" : "fp32",
                 g.model == LBM_CS ? cs_tile_tx(best_tile) : fd_tile_tx(best_tile),
                 g.model == LBM_CS ? cs_tile_ty(best_tile) : fd_tile_ty(best_tile), g.grid, best / trial_steps);
        rep += b;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    invalidate_graph();
    if (report) *report = rep;
    return LBM_OK;
}

}  // namespace lbm
