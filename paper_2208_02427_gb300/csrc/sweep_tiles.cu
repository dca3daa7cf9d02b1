// sweep_tiles.cu -- several point sweeps in one launch, on tiles in shared memory.
//
// A small grid is bound by launches, not by its sweeps: a colour pass over 513 x 385 points is 0.8 us of
// FP64 arithmetic in a launch of 2.0 us. Here a CTA loads its tile with a halo of one
// point per pass, runs the passes of `sweeps` sweeps in shared memory with a CTA barrier between them,
// and writes its own points to the other buffer. Each pass covers one halo point less than the one
// before, so every value is the one that the passes over the whole grid would have left: the same
// expression of the same operands, bit for bit. The halo costs arithmetic (a 37 x 39 tile does 1.3 times its
// own points over three red-black sweeps), so the number of sweeps and the tile follow from the grid
// (plan_sweep_tiles). What is left beside the FP64 work: a launch and the window's load and store, 1.4 us
// or more, and about 0.4 us a pass (a point's chain of FP64 operations of 71 cycles each, the barrier, the
// warps' uneven last round).
#include <algorithm>
#include <cmath>

#include "lap_device.cuh"
#include "lap_internal.cuh"
#include "vcycle_arith.cuh"

namespace lap {

namespace {

constexpr int ST_THREADS = 512;
constexpr size_t ST_SMEM_MAX = 224 * 1024;
// The cost model of plan_sweep_tiles, in SM cycles beside the FP64 work: a one-pass launch (the walks along
// diagonals take longer to drain), a tile launch, a window point's load and store, and a pass's latency,
// barrier and uneven last round. Fitted to times per sweep from 65^2 to 4097^2 points.
constexpr double PASS_CYCLES = 2600, DIAG_PASS_CYCLES = 3600;
constexpr double TILE_CYCLES = 2900, TILE_POINT_CYCLES = 0.4, TILE_PASS_CYCLES = 900;

__device__ __forceinline__ void copy8(double* smem, const double* global)
{
    const unsigned dst = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(global) : "memory");
}

struct SweepCoef {
    double b2, inv_d;
    int shift;
    double w, omw;
};

// One point from the tile `a` (row pitch W): the expression of the one-pass kernels.
template <int KIND, bool UNIT, bool POW2, bool DIAG>
__device__ __forceinline__ double swept(const FmaOps& o, const double* c, int W, const SweepCoef& k)
{
    const double s = DIAG ? fadd(o, fadd(o, c[-1], c[-W]), fadd(o, c[1], c[W]))
                          : neighbour_sum<UNIT>(o, c[-1], c[1], c[-W], c[W], k.b2);
    const double g = times_inv_d<POW2>(o, s, k.inv_d, k.shift);
    return KIND == SWEEP_SOR ? __fma_rn(k.w, g, fmul(o, k.omw, *c)) : g;
}

// Points that a tile's window reaches past its own in a launch of `passes` passes. No pass is a copy: the ring
// beside the tile all the same.
__host__ __device__ constexpr int window_halo(int passes) { return passes > 1 ? passes : 1; }

// The tile of interior columns [x0, x1) and rows [y0, y1) through `passes` passes (two colours a sweep, or
// one for Jacobi), in -> out. ring: the ring points beside the tile are copied along, so that a second buffer
// needs no preparation (the caller's ring is never written). sm: (x1 - x0 + 2 h) (y1 - y0 + 2 h) doubles, h = window_halo(passes), twice that for Jacobi.
template <int KIND, bool UNIT, bool POW2, bool DIAG>
__device__ __forceinline__ void sweep_tile(const FmaOps& o, const double* __restrict__ in, double* __restrict__ out,
                                           int m, int n, int64_t pitch, int64_t pitch_out, int x0, int x1, int y0,
                                           int y1, int passes, bool ring, const SweepCoef& k, double* sm)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int h = window_halo(passes);
    const int X0 = max(0, x0 - h), X1 = min(m, x1 + h);
    const int Y0 = max(0, y0 - h), Y1 = min(n, y1 + h);
    const int W = X1 - X0, H = Y1 - Y0;
    for (int r = wid; r < H; r += nw) {
        const double* src = in + (int64_t)(Y0 + r) * pitch + X0;
        for (int c = lane; c < W; c += 32) copy8(sm + r * W + c, src + c);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    double* a = sm;
    double* b = sm + W * H;
    if (KIND == SWEEP_JACOBI) {
        // the ring, which no pass writes, in the second buffer too
        for (int t = threadIdx.x; t < W; t += blockDim.x) {
            b[t] = a[t];
            b[(H - 1) * W + t] = a[(H - 1) * W + t];
        }
        for (int t = threadIdx.x; t < H; t += blockDim.x) {
            b[t * W] = a[t * W];
            b[t * W + W - 1] = a[t * W + W - 1];
        }
        __syncthreads();
    }
    // A pass's region [ia, ib) x [ja, jb) of the window, `per` of its points to a row; thread t takes points
    // t, t + blockDim, .. row by row: first (r, c), then (dr, dc) on. The quotients from the FP32 divide are
    // exact: (t + 1/2) / per is at least 1 / (2 per) away from a whole number. Taken before the barrier that
    // ends the pass before, so that this arithmetic runs beside that pass's FP64 chains.
    int ia, ib, ja, rows, per, r, c, dr, dc;
    auto region = [&](int p) {
        ia = X0 == 0 ? 1 : p + 1;
        ib = W - (X1 == m ? 1 : p + 1);
        ja = Y0 == 0 ? 1 : p + 1;
        rows = H - (Y1 == n ? 1 : p + 1) - ja;
        per = KIND == SWEEP_JACOBI ? ib - ia : (ib - ia + 1) / 2;
        const float inv = __fdividef(1.0f, (float)per);
        r = (int)(((float)threadIdx.x + 0.5f) * inv);
        c = threadIdx.x - r * per;
        dr = (int)(((float)blockDim.x + 0.5f) * inv);
        dc = blockDim.x - dr * per;
    };
    region(0);
    for (int p = 0; p < passes; ++p) {
        double* dst = KIND == SWEEP_JACOBI ? b : a;
        while (r < rows) {
            const int j = ja + r;
            const int i = ia + (KIND == SWEEP_JACOBI ? c : ((ia + X0 + j + Y0 + p) & 1) + 2 * c);
            const int at = j * W + i;
            if (KIND == SWEEP_JACOBI || i < ib) dst[at] = swept<KIND, UNIT, POW2, DIAG>(o, a + at, W, k);
            c += dc;
            r += dr;
            if (c >= per) {
                c -= per;
                ++r;
            }
        }
        region(p + 1 < passes ? p + 1 : p);
        __syncthreads();
        if (KIND == SWEEP_JACOBI) {
            double* t = a;
            a = b;
            b = t;
        }
    }
    const int sx0 = ring && x0 == 1 ? 0 : x0, sx1 = ring && x1 == m - 1 ? m : x1;
    const int sy0 = ring && y0 == 1 ? 0 : y0, sy1 = ring && y1 == n - 1 ? n : y1;
    for (int j = sy0 + wid; j < sy1; j += nw)
        for (int i = sx0 + lane; i < sx1; i += 32) out[(int64_t)j * pitch_out + i] = a[(j - Y0) * W + (i - X0)];
}

// Tile (blockIdx.x, blockIdx.y) of gridDim.x x gridDim.y equal parts of the interior.
template <int KIND, bool UNIT, bool POW2, bool DIAG>
__global__ void __launch_bounds__(ST_THREADS)
    sweep_tiles_kernel(const double* __restrict__ in, double* __restrict__ out, int m, int n, int64_t pitch,
                       int64_t pitch_out, int passes, int ring, SweepCoef k, const double* __restrict__ wslot)
{
    after_prior();
    extern __shared__ double sm[];
    const FmaOps o = load_fma_ops();
    if (KIND == SWEEP_SOR) {
        k.w = wslot[0];
        k.omw = wslot[1];
    }
    if (!UNIT) k.b2 = in_reg(o, k.b2);
    if (!POW2) k.inv_d = in_reg(o, k.inv_d);
    const int x0 = 1 + (int)((int64_t)blockIdx.x * (m - 2) / gridDim.x);
    const int x1 = 1 + (int)((int64_t)(blockIdx.x + 1) * (m - 2) / gridDim.x);
    const int y0 = 1 + (int)((int64_t)blockIdx.y * (n - 2) / gridDim.y);
    const int y1 = 1 + (int)((int64_t)(blockIdx.y + 1) * (n - 2) / gridDim.y);
    sweep_tile<KIND, UNIT, POW2, DIAG>(o, in, out, m, n, pitch, pitch_out, x0, x1, y0, y1, passes,
                                       ring != 0, k, sm);
}

// Launch `k` of `launches` over the tiles of many fields (SOR, each field's own factor and spacing): an even
// launch takes a field to its second buffer and an odd one back, each with its share of the field's sweeps,
// at times none (a copy). Bound by FP64 and, between its tiles' barriers, by latency: three CTAs to a
// multiprocessor (40 registers) against two: 108.6 against 112 ms on the burst below.
__global__ void __launch_bounds__(ST_THREADS, 3)
    b_sweep_tiles_kernel(const SweepTileItem* __restrict__ items, const int* __restrict__ active, int k, int launches)
{
    after_prior();
    extern __shared__ double sm[];
    const FmaOps o = load_fma_ops();
    const SweepTileItem it = items[blockIdx.x];
    if (!active[it.problem]) return;
    const int passes = 2 * (it.sweeps / launches + (k < it.sweeps % launches ? 1 : 0));
    const bool back = k & 1;
    SweepCoef c{it.b2, it.inv_d, it.inv_d_shift, in_reg(o, it.w), in_reg(o, it.omw)};
    auto run = [&](auto U, auto P) {
        if (!decltype(U)::value) c.b2 = in_reg(o, c.b2);
        if (!decltype(P)::value) c.inv_d = in_reg(o, c.inv_d);
        sweep_tile<SWEEP_SOR, decltype(U)::value, decltype(P)::value, false>(
            o, back ? it.other : it.u, back ? it.u : it.other, it.m, it.n, back ? it.pitch_other : it.pitch,
            back ? it.pitch : it.pitch_other, it.x0, it.x1, it.y0, it.y1, passes, !back, c, sm);
    };
    on_flag(it.unit_beta != 0, [&](auto U) { on_flag(it.inv_d_shift > 0, [&](auto P) { run(U, P); }); });
}

template <class F>
cudaError_t on_sweep_kernel(const Coef& c, int kind, bool diag, F&& f)
{
    const bool pow2 = c.inv_d_shift > 0;
    if (kind == SWEEP_JACOBI) {
        if (c.unit_beta) return pow2 ? f(sweep_tiles_kernel<SWEEP_JACOBI, true, true, false>)
                                     : f(sweep_tiles_kernel<SWEEP_JACOBI, true, false, false>);
        return pow2 ? f(sweep_tiles_kernel<SWEEP_JACOBI, false, true, false>)
                    : f(sweep_tiles_kernel<SWEEP_JACOBI, false, false, false>);
    }
    if (kind == SWEEP_SOR) {
        if (diag) return f(sweep_tiles_kernel<SWEEP_SOR, true, true, true>);
        if (c.unit_beta) return pow2 ? f(sweep_tiles_kernel<SWEEP_SOR, true, true, false>)
                                     : f(sweep_tiles_kernel<SWEEP_SOR, true, false, false>);
        return pow2 ? f(sweep_tiles_kernel<SWEEP_SOR, false, true, false>)
                    : f(sweep_tiles_kernel<SWEEP_SOR, false, false, false>);
    }
    if (diag) return f(sweep_tiles_kernel<SWEEP_GS, true, true, true>);
    if (c.unit_beta) return pow2 ? f(sweep_tiles_kernel<SWEEP_GS, true, true, false>)
                                 : f(sweep_tiles_kernel<SWEEP_GS, true, false, false>);
    return pow2 ? f(sweep_tiles_kernel<SWEEP_GS, false, true, false>)
                : f(sweep_tiles_kernel<SWEEP_GS, false, false, false>);
}

int halo(int kind, int sweeps) { return kind == SWEEP_JACOBI ? sweeps : 2 * sweeps; }

}  // namespace

// At most one tile per multiprocessor, nearly square, and as many sweeps per launch as cost least; none
// where the one-pass kernels are within 2%. Measured per sweep (one pass per launch / tiles), SOR in the
// paper's order: 129^2 2.66 / 1.79 us, 257^2 2.98 / 2.40, 513 x 385 4.02 / 3.87, 700^2 6.92 / 6.64, 850^2
// 8.93 / 9.07, 1000^2 11.1 / 11.7; paired along diagonals 5.20 / 1.78, 5.33 / 2.38, 5.68 / 3.88, 7.40 / 6.64, 9.01 /
// 9.06, 10.8 / 11.7; Gauss-Seidel 700^2 5.02 / 4.84, 850^2 6.25 / 6.40; Jacobi 129^2 1.42 / 0.96, 257^2 1.64 / 1.38,
// 513 x 385 2.26 / 2.22, 850^2 5.07 / 5.25. Two or three smaller tiles per multiprocessor hide a tile's load but
// have more halo: equal or slower.
SweepTiles plan_sweep_tiles(int m, int n, const Coef& c, int kind, bool diag, int sms)
{
    SweepTiles best;
    const int colours = kind == SWEEP_JACOBI ? 1 : 2;
    const double ops = 3.0 + (c.inv_d_shift > 0 ? 0 : 1) + (kind == SWEEP_SOR ? 2 : 0);
    // per sweep; an FP64 operation takes half a cycle of an SM
    double least = colours * (diag ? DIAG_PASS_CYCLES : PASS_CYCLES) +
                   1.07 * (m - 2) * (double)(n - 2) * (ops - (diag ? 1 : 0)) / 2 / sms;
    least *= 0.98;
    const int near = (int)std::min(std::sqrt((double)sms * (m - 2) / (n - 2)), (double)sms);
    for (int sweeps = 1; sweeps <= 8; ++sweeps) {
        const int h = halo(kind, sweeps);
        for (int tx = std::max(1, near - 2); tx <= std::min({sms, m - 2, near + 3}); ++tx) {
            const int ty = std::min(sms / tx, n - 2);
            const int64_t tw = (m - 2 + tx - 1) / tx, th = (n - 2 + ty - 1) / ty;
            const int64_t window = (tw + 2 * h) * (th + 2 * h);
            if (window * 8 * (kind == SWEEP_JACOBI ? 2 : 1) > (int64_t)ST_SMEM_MAX) continue;
            // points of the h passes: (tw + 2a)(th + 2a) for a = 0 .. h - 1, one colour of them
            const double sum = (double)h * tw * th + (double)(tw + th) * h * (h - 1) + 2.0 / 3.0 * h * (h - 1) * (2 * h - 1);
            const double cost =
                (TILE_CYCLES + window * TILE_POINT_CYCLES + h * TILE_PASS_CYCLES + sum / colours * ops / 2) / sweeps;
            if (cost < least) {
                least = cost;
                best = SweepTiles{sweeps, tx, ty};
            }
        }
    }
    return best;
}

cudaError_t prepare_sweep_tiles(const Coef& c, int kind, bool diag)
{
    return on_sweep_kernel(c, kind, diag, [](auto* kernel) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ST_SMEM_MAX);
    });
}

cudaError_t launch_sweep_tiles(const Field& in, double* out, int64_t pitch_out, const Coef& c, const SweepTiles& t,
                               int kind, bool diag, int sweeps, bool ring, const double* wslot, cudaStream_t s)
{
    const int passes = halo(kind, sweeps), h = window_halo(passes);
    const int tw = (in.m - 2 + t.tx - 1) / t.tx, th = (in.n - 2 + t.ty - 1) / t.ty;
    const size_t bytes = (size_t)(tw + 2 * h) * (th + 2 * h) * 8 * (kind == SWEEP_JACOBI ? 2 : 1);
    const SweepCoef k{c.b2, c.inv_d, c.inv_d_shift, 1.0, 0.0};
    const cudaError_t e = on_sweep_kernel(c, kind, diag, [&](auto* kernel) {
        launch_after(kernel, dim3(t.tx, t.ty), ST_THREADS, bytes, s, in.p, out, in.m, in.n, in.pitch, pitch_out,
                     passes, ring ? 1 : 0, k, wslot);
        return cudaGetLastError();
    });
    note_launch();
    return e;
}

// Tile sides and sweeps per launch that cost least for SOR fields of m[k] x n[k] points, by the model of
// plan_sweep_tiles with the tiles in as many rounds as it takes. Sides are tried around those that give
// one, two or three tiles per multiprocessor (or as many as shared memory needs), upright and flat.
// Per colour pass of a step of 50 sweeps, one pass per launch / tiles: one field of 33^2 points 4.0 / 1.4 us,
// 257^2 5.0 / 2.5, 513^2 7.2 / 3.8, 1025^2 11.5 / 7.8, four of 1025^2 26.5 / 23.6 (FP64 alone 16.8). A burst of
// 48 requests (sides 33..1025, half of them SOR): 125.6 / 108.6 ms.
// Fields of one size count once, sides past the widest field's are as good as its own, and a pair of sides is
// only worked out where a lower bound of its cost (no partial tiles, no partial last round) beats the best
// cost so far: a step plans on the host with the device idle. 1000 fields of different sizes take 0.28 ms, every pair
// of sides over every field 1.16 (one host core).
BatchSweepPlan plan_batch_sweeps(const std::vector<std::pair<int, int>>& fields, int sms)
{
    BatchSweepPlan best;
    double least = 1e300;
    const int most_side = 148;
    struct Group {
        double m, n, count;
    };
    std::vector<Group> groups;
    double points = 0, halves = 0, widest = 1, tallest = 1;
    {
        std::vector<std::pair<int, int>> sorted(fields);
        std::sort(sorted.begin(), sorted.end());
        for (size_t k = 0; k < sorted.size(); ++k) {
            if (k > 0 && sorted[k] == sorted[k - 1]) groups.back().count += 1;
            else groups.push_back({(double)(sorted[k].first - 2), (double)(sorted[k].second - 2), 1.0});
        }
    }
    for (const Group& g : groups) {
        points += g.count * g.m * g.n;
        halves += g.count * (g.m + g.n);
        widest = std::max(widest, g.m);
        tallest = std::max(tallest, g.n);
    }
    // cycles of `t` tiles with `a` points and half rims of `r` in all, h passes a launch: the FP64 work of
    // their passes and their windows
    auto cycles = [](int h, double t, double a, double r) {
        const double sum = h * a + r * h * (h - 1) + t * 2.0 / 3.0 * h * (h - 1) * (2 * h - 1);
        return sum / 2 * 5 / 2 + (a + 2 * h * r + t * 4.0 * h * h) * TILE_POINT_CYCLES;
    };
    // the cost for `sweeps` a launch, given the busiest multiprocessor's cycles (1e300: no room)
    auto cost = [](int sx, int sy, int sweeps, double busy) {
        if ((int64_t)(sx + 4 * sweeps) * (sy + 4 * sweeps) * 8 > (int64_t)ST_SMEM_MAX) return 1e300;
        return (TILE_CYCLES + 2 * sweeps * TILE_PASS_CYCLES + busy) / sweeps;
    };
    struct Sides {
        double bound;
        int sx, sy, order;  // of sides that cost the same, the first tried: the smaller windows
    };
    std::vector<Sides> tried;
    std::vector<char> seen((most_side + 1) * (most_side + 1), 0);
    const int fewest = std::max(1, (int)std::ceil(points / ((double)sms * most_side * most_side)));
    for (int per_sm = fewest; per_sm < fewest + 3; ++per_sm) {
        const double even_side = std::sqrt(points / ((double)sms * per_sm));
        for (double factor = 0.94; factor < 1.6; factor *= 1.02) {
            for (double flat : {1.0, 0.87, 0.75}) {
                const int side = (int)std::min<double>(most_side, std::max(6.0, even_side * factor));
                const int sx = (int)std::min<double>(side, widest), sy = (int)std::min(std::max(6.0, side * flat), tallest);
                char& known = seen[sx * (most_side + 1) + sy];
                if (known) continue;
                known = 1;
                const double tiles = std::max((double)fields.size(), points / (sx * sy));
                const double rim = std::max(halves, points / sx + points / sy);
                Sides t{1e300, sx, sy, (int)tried.size()};
                for (int sweeps = 1; sweeps <= 6; ++sweeps)
                    t.bound = std::min(t.bound, cost(sx, sy, sweeps, cycles(2 * sweeps, tiles, points, rim) / sms));
                tried.push_back(t);
            }
        }
    }
    std::sort(tried.begin(), tried.end(), [](const Sides& a, const Sides& b) { return a.bound < b.bound; });
    int order = 0;
    for (const Sides& t : tried) {
        if (t.bound > least) break;
        double tiles = 0, rim = 0, tw1 = 1, th1 = 1;
        const double ix = 1.0 / t.sx, iy = 1.0 / t.sy;
        for (const Group& g : groups) {
            // parts of a side, rounded up (the half keeps the product off whole numbers)
            const double tx = 1 + (int)((g.m - 0.5) * ix), ty = 1 + (int)((g.n - 0.5) * iy);
            tiles += g.count * tx * ty;
            rim += g.count * (g.m * ty + g.n * tx);
            if (g.m * g.n > tw1 * th1 * (tx * ty)) tw1 = g.m / tx, th1 = g.n / ty;
        }
        const double rounds = std::ceil(tiles / sms);
        for (int sweeps = 1; sweeps <= 6; ++sweeps) {
            const int h = 2 * sweeps;
            const double busy = std::max(cycles(h, 1, tw1 * th1, tw1 + th1), cycles(h, tiles, points, rim) / tiles * rounds);
            const double c = cost(t.sx, t.sy, sweeps, busy);
            if (c < least || (c == least && t.order < order)) {
                least = c;
                order = t.order;
                best = BatchSweepPlan{sweeps, t.sx, t.sy};
            }
        }
    }
    return best;
}

void add_sweep_tiles(std::vector<SweepTileItem>& items, SweepTileItem it, const BatchSweepPlan& plan)
{
    const int tx = (it.m - 2 + plan.sx - 1) / plan.sx, ty = (it.n - 2 + plan.sy - 1) / plan.sy;
    for (int y = 0; y < ty; ++y)
        for (int x = 0; x < tx; ++x) {
            it.x0 = 1 + (int)((int64_t)x * (it.m - 2) / tx);
            it.x1 = 1 + (int)((int64_t)(x + 1) * (it.m - 2) / tx);
            it.y0 = 1 + (int)((int64_t)y * (it.n - 2) / ty);
            it.y1 = 1 + (int)((int64_t)(y + 1) * (it.n - 2) / ty);
            items.push_back(it);
        }
}

cudaError_t launch_b_sweep_tiles(const SweepTileItem* items, int count, const BatchSweepPlan& plan, const int* active,
                                 int k, int launches, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    const size_t bytes = (size_t)(plan.sx + 4 * plan.sweeps) * (plan.sy + 4 * plan.sweeps) * 8;
    if (k == 0) {
        const cudaError_t e = cudaFuncSetAttribute(b_sweep_tiles_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)ST_SMEM_MAX);
        if (e != cudaSuccess) return e;
    }
    launch_after(b_sweep_tiles_kernel, count, ST_THREADS, bytes, s, items, active, k, launches);
    note_launch();
    return cudaGetLastError();
}

}  // namespace lap
