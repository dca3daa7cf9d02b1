// lap_host.cuh -- host-side internals shared by the C-ABI sources of liblaplace.so
// (lap_api.cu: handles, single-grid solves and component calls; lap_batched.cu: many grids
// at once; lap_server.cu: the serving loop). Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <deque>
#include <map>
#include <memory>
#include <mutex>
#include <stdexcept>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/laplace.h"
#include "lap_internal.cuh"

namespace lap {

int64_t launches_now();
void add_launches(int64_t k);

// One launch configuration of a batched V-cycle; none of its choices changes a computed value.
struct BatchConfig {
    int tail;   // small-level tail size (-1: none)
    int tiles;  // FP32 levels of the mixed solver: 0 = one kernel per pass (temporal depth 1),
                // 1..FUSED32_VARIANTS = a level's whole descent / ascent per tile load (depth nu)
                // with that tile variant (CTA size and region rows), FUSED32_STREAMS = row streams
    int item;   // interior points per work item of the per-pass kernels
    int persist;  // 1: every phase a persistent launch (resident CTAs claim its items), 0: one CTA per item
    bool operator==(const BatchConfig& o) const
    {
        return tail == o.tail && tiles == o.tiles && item == o.item && persist == o.persist;
    }
};

extern thread_local std::string t_last_error;

struct Error {
    int code;
    std::string msg;
};

[[noreturn]] inline void fail(int code, const std::string& msg) { throw Error{code, msg}; }

inline void ck(cudaError_t e, const char* what)
{
    if (e != cudaSuccess) fail(LAP_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

template <class F>
int guarded(F&& body)
{
    try {
        body();
        return LAP_OK;
    } catch (const Error& e) {
        t_last_error = e.msg;
        return e.code;
    } catch (const std::bad_alloc&) {
        t_last_error = "host allocation failed";
        return LAP_ENOMEM;
    } catch (...) {
        t_last_error = "unexpected internal error";
        return LAP_ECUDA;
    }
}

inline int64_t round_up(int64_t v, int64_t a) { return (v + a - 1) / a * a; }

// A batched solve's plan kept in the handle for the next call on the same batch (defined in
// lap_batched.cu; destroyed with the handle or when another batch or call takes the arena).
struct BatchCacheBase {
    virtual ~BatchCacheBase() = default;
};

// Host-side copy of a line-solver table set plus its device allocation.
struct LineEntry {
    LineTables t;
    double* dev = nullptr;
    size_t bytes = 0;
};

struct CoarseEntry {
    double* dev = nullptr;
    size_t bytes = 0;
};

}  // namespace lap

struct lap_handle_s {
    int device = 0;
    size_t budget = 0;    // 0 = unlimited
    size_t held = 0;      // bytes of device memory held (arena + tables)
    double* arena = nullptr;
    size_t arena_bytes = 0;
    uint64_t arena_epoch = 0;  // counts the calls that carved the arena (arena())
    std::unique_ptr<lap::BatchCacheBase> batch_cache;  // the last batched solve's plan
    double* pinned = nullptr;  // 8 doubles of pinned host memory for results
    std::map<std::tuple<int, double, double, double, int, int>, lap::LineEntry> lines;
    std::map<std::tuple<int, int, double>, lap::CoarseEntry> coarse;
    // CUDA graphs of whole check periods (the iterations between two stopping tests),
    // keyed by every pointer and parameter baked into them; replayed on the caller's stream
    bool use_graphs = true;
    cudaStream_t capture = nullptr;
    std::map<std::string, std::pair<cudaGraphExec_t, int64_t>> graphs;  // exec, kernels
    lap::BatchConfig last_batch{0, 0, 0, 0};  // the configuration the last batched cycle ran
    // y-line scratch of line relaxation: forward-elimination values and chunk ends (grown on
    // demand)
    double* lscratch = nullptr;
    size_t lscratch_bytes = 0;
    void* spare = nullptr;  // second field of the tiled sweeps; given back when memory is short
    size_t spare_bytes = 0;
    // x-line sweeps: error word, item counter and row flags; one block of at least 1 MiB,
    // allocated on first use and grown only for more than 262,140 lines
    unsigned* lsync = nullptr;
    size_t lsync_bytes = 0;
    // device copy of the field of lap_solve_host (grown on demand)
    double* hfield = nullptr;
    size_t hfield_bytes = 0;
};

namespace lap {

void set_device(lap_handle h);
void* dev_alloc(lap_handle h, size_t bytes);
void dev_free(lap_handle h, void* p, size_t bytes);
void drop_graphs(lap_handle h);
// Scratch for one call: grows (never shrinks) the handle's arena.
double* arena(lap_handle h, size_t bytes);
// The handle's spare buffer of at least `bytes`, or null where the budget or the device has no room for
// it, or it would be more than SPARE_MAX: a call that can do without takes its other path. (The rows of the
// tallest grid of lines, 1024 unknowns to a row and 16383 rows, come to SPARE_MAX; tiles pay up to about a million points.)
constexpr size_t SPARE_MAX = (size_t)64 << 20;
double* spare(lap_handle h, size_t bytes);

// Carves aligned sub-buffers out of a byte range.
struct Carver {
    char* base;
    size_t off = 0;
    explicit Carver(void* b) : base((char*)b) {}
    template <class T>
    T* take(size_t count)
    {
        off = (size_t)round_up((int64_t)off, 256);
        T* p = (T*)(base + off);
        off += count * sizeof(T);
        return p;
    }
};
// The same carving sequence without memory, to size the arena first.
struct Sizer {
    size_t off = 0;
    template <class T>
    T* take(size_t count)
    {
        off = (size_t)round_up((int64_t)off, 256) + count * sizeof(T);
        return nullptr;
    }
};

void check_grid(const lap_grid* g);
void check_device_ptr(lap_handle h, const void* p, const char* what, bool allow_null = false);
void check_params(const lap_params* p);

// line relaxation: cached tables of a line length and coefficients; the tables, coefficients
// and scratch of a half sweep (allocating only on a shape's first use); one zebra half sweep
constexpr int LINE_MIN_CHUNK = 16;
constexpr int LINE_Y_MIN_CHUNK = 4;
const LineTables& line_tables(lap_handle h, int N, double alpha, double delta, double wc,
                              int max_chunks = LINE_MAX_CHUNKS, int min_chunk = LINE_MIN_CHUNK);
const LineTables& line_setup(lap_handle h, const Field& f, const Coef& c, double w, int form,
                             int direction, LineCoefs* k, double** scratch, bool threads = false);
double* line_rows(lap_handle h, const Field& f, const Coef& c, double w, int form);
void line_half_sweep(lap_handle h, const Field& f, const Coef& c, double w, int form,
                     int direction, cudaStream_t s, double* rows = nullptr);

// the coarsest level's 5-point matrix, inverted once per shape (transposed, on the device)
constexpr int COARSE_MAX_UNKNOWNS = 1024;
const double* coarse_inverse(lap_handle h, int m, int n, double b2, double d);
int mg_level_count(int m, int n, int coarsest_min, int max_levels);


// ---- V-cycles over many problems (lap_batched.cu, lap_server.cu) ----
// Interior points per work item (rows are not split) of the norm, update and server lists. A batch's
// level passes have items by its size (batch_config). Measured on the 4096-grid batch (sides
// 33..513, V(2,2) to 1e-10) with all lists alike: FP64 145 / 140 / 140 / 145 ms at 2048 / 8192 / 16384 /
// 32768 points, the mixed solver 74 / 71 / 69 / 68 ms.
constexpr int BATCH_ITEM_POINTS = 8192;
void add_items(std::vector<BatchItem>& items, int level_index, int m, int n,
               int points = BATCH_ITEM_POINTS, bool red = false, int unit = 1);

// Per-level work lists of one V-cycle over a set of problems: [first, count) into the items
// (fine, all, coarse) or into the tail jobs (tail).
struct LevelLists {
    std::vector<std::pair<int, int>> fine, all, coarse, tail;
    std::vector<std::pair<int, int>> tiles;  // FP32 tile items of the fine lists (fused cycle)
    std::vector<std::pair<int, int>> sdown, sup;  // the same as pieces of row streams
    std::pair<int, int> upd0{0, 0};  // fused: level-0 items of the problems without level-0 tiles
    bool fused = false;
    int tile_variant = 1;  // the fused FP32 levels' tile variant, or FUSED32_STREAMS
    unsigned* claim = nullptr;  // non-null: every launch persistent, claiming items here (BatchList)
    int levels = 0;
    int max_coarse = 0;
    // shared memory of the tail jobs of a level in FP64 and FP32 (smem_tail_kernel; 0: some job does
    // not fit, b_tail_kernel)
    std::vector<size_t> tail64, tail32;
};

// First level of a problem that the small-level tail runs (both sides <= tail_size), or
// nlev when it has none.
int tail_start(const BatchLevel<double>* lv, int nlev, int tail_size);

// Lists of one V-cycle over problems `who`: problem q owns levels base[q] .. base[q] +
// nlev[q] - 1 of lv. Levels above a problem's tail go through item lists, the tail is one job.
// With tiles and streams, the fine levels also get the items of the fused FP32 descent/ascent: tile
// items, or with tile_variant FUSED32_STREAMS pieces of row streams (and level-0 tile items too when
// level0_tiles: the descents of a later inner cycle do not start from zero).
void build_lists(LevelLists& L, std::vector<BatchItem>& items, std::vector<TailJob>& jobs,
                 const std::vector<int>& who, const std::vector<int>& base,
                 const std::vector<int>& nlev, const std::vector<BatchLevel<double>>& lv,
                 int tail_size, std::vector<TileItem>* tiles = nullptr,
                 std::vector<StreamItem>* streams = nullptr, int nu1 = 0, int nu2 = 0,
                 int tile_variant = 1, bool level0_tiles = false, int item_points = BATCH_ITEM_POINTS);

// The tail jobs of level l.
template <class T>
void enqueue_tail(const LevelLists& L, int l, const BatchLevel<T>* lv, const int* active, const TailJob* jobs,
                  const lap_params& p, double smoother_w, cudaStream_t st)
{
    const bool gs = smoother_w == 1.0;
    SmemTail plan;
    plan.bytes = (sizeof(T) == 8 ? L.tail64 : L.tail32)[l];
    if (plan.bytes)
        ck(launch_smem_tail(jobs + L.tail[l].first, L.tail[l].second, lv, active, p.nu1, p.nu2, gs, smoother_w, plan,
                            st, L.claim),
           "batched tail");
    else
        ck(launch_b_tail(jobs + L.tail[l].first, L.tail[l].second, lv, active, p.nu1, p.nu2, gs, smoother_w,
                         L.max_coarse, st, L.claim),
           "batched tail");
}

// One V-cycle over every active problem of L: descend (coarsest solves and tails start when
// the descent reaches a problem's coarsest or tail level), then ascend; each problem sees
// its own V-cycle.
template <class ListFn, class T>
void enqueue_vcycle(ListFn list, const LevelLists& L, const BatchLevel<T>* lv, const int* active,
                    const TailJob* jobs, const lap_params& p, double smoother_w, cudaStream_t st)
{
    const bool gs = smoother_w == 1.0;
    for (int l = 0; l < L.levels; ++l) {
        ck(launch_b_coarse(list(L.coarse[l]), lv, active, L.max_coarse, st), "batched coarse");
        enqueue_tail(L, l, lv, active, jobs, p, smoother_w, st);
        if (l == L.levels - 1) break;
        // below level 0 the restriction has done the first red pass
        for (int k = l > 0 && gs ? 1 : 0; k < 2 * p.nu1; ++k)
            ck(launch_b_rb(list(L.fine[l]), lv, active, k & 1, gs, smoother_w, st), "batched smoother");
        const bool after_gs = gs && p.nu1 > 0;
        ck(launch_b_defect(list(L.fine[l]), lv, active, st, after_gs), "batched defect");
        ck(launch_b_restrict(list(L.all[l + 1]), lv, active, st, after_gs), "batched restrict");
    }
    for (int l = L.levels - 2; l >= 0; --l) {
        ck(launch_b_prolong(list(L.fine[l]), lv, active, st, gs && p.nu2 > 0), "batched prolong");
        for (int k = 0; k < p.nu2; ++k)
            for (int colour = 0; colour < 2; ++colour)
                ck(launch_b_rb(list(L.fine[l]), lv, active, colour, gs, smoother_w, st), "batched smoother");
    }
}

// The FP32 V-cycle with each fine level's descent and ascent as one launch of tiles or row streams
// over all problems (first: the level-0 corrections start at zero).
// fold64 (nullable): the level-0 ascent adds its result to these FP64 fields (psi += e).
template <class ListFn>
void enqueue_vcycle32_fused(ListFn list, const LevelLists& L, const BatchLevel<float>* lv,
                            const int* active, const TailJob* jobs, const TileItem* tiles,
                            const StreamItem* streams, const lap_params& p, double smoother_w, bool first,
                            cudaStream_t st, const BatchLevel<double>* fold64 = nullptr)
{
    const bool gs = smoother_w == 1.0, rows = L.tile_variant == FUSED32_STREAMS;
    const int variant = rows ? 1 : L.tile_variant;
    for (int l = 0; l < L.levels; ++l) {
        ck(launch_b_coarse(list(L.coarse[l]), lv, active, L.max_coarse, st), "batched coarse");
        enqueue_tail(L, l, lv, active, jobs, p, smoother_w, st);
        if (l == L.levels - 1) break;
        if (rows && (l > 0 || first))
            ck(launch_b_stream_down(streams + L.sdown[l].first, L.sdown[l].second, lv, active, p.nu1, gs,
                                    smoother_w, st),
               "batched descent");
        else
            ck(launch_b_down32(tiles + L.tiles[l].first, L.tiles[l].second, lv, active, p.nu1,
                               l > 0 || first, gs, smoother_w, st, variant, L.claim),
               "batched descent");
    }
    for (int l = L.levels - 2; l >= 0; --l) {
        if (rows)
            ck(launch_b_stream_up(streams + L.sup[l].first, L.sup[l].second, lv, active, p.nu2, gs, smoother_w,
                                  st, l == 0 ? fold64 : nullptr),
               "batched ascent");
        else
            ck(launch_b_up32(tiles + L.tiles[l].first, L.tiles[l].second, lv, active, p.nu2, gs,
                             smoother_w, st, l == 0 ? fold64 : nullptr, variant, L.claim),
               "batched ascent");
    }
}

}  // namespace lap
