// The server's tile plan against the search it stands for: every pair of sides tried with every field, in plain
// loops. Prints, for sets of many kinds, the largest ratio of the plan's cost to the search's, then the host times
// of both for 1000 fields of different sizes in microseconds.
#include <chrono>
#include <cstdio>
#include <random>

#include "sweep_tiles.cu"

namespace lap {
void note_launch() {}
}  // namespace lap
using namespace lap;
using Fields = std::vector<std::pair<int, int>>;

// The cost model: cycles per sweep of fields on tiles of at most sx x sy points (1e300: no room).
static double cost_of(const Fields& fields, int sms, int sweeps, int sx, int sy)
{
    const int h = 2 * sweeps;
    if ((int64_t)(sx + 2 * h) * (sy + 2 * h) * 8 > (int64_t)ST_SMEM_MAX) return 1e300;
    double tiles = 0, rim = 0, points = 0, tw1 = 1, th1 = 1;
    for (const auto& f : fields) {
        const int tx = (f.first - 2 + sx - 1) / sx, ty = (f.second - 2 + sy - 1) / sy;
        const double tw = (double)(f.first - 2) / tx, th = (double)(f.second - 2) / ty;
        tiles += (double)tx * ty;
        rim += (double)tx * ty * (tw + th);
        points += (double)(f.first - 2) * (f.second - 2);
        if (tw * th > tw1 * th1) tw1 = tw, th1 = th;
    }
    auto cycles = [&](double t, double a, double r) {
        const double sum = h * a + r * h * (h - 1) + t * 2.0 / 3.0 * h * (h - 1) * (2 * h - 1);
        return sum / 2 * 5 / 2 + (a + 2 * h * r + t * 4.0 * h * h) * TILE_POINT_CYCLES;
    };
    const double busy = std::max(cycles(1, tw1 * th1, tw1 + th1), cycles(tiles, points, rim) / tiles * std::ceil(tiles / sms));
    return (TILE_CYCLES + h * TILE_PASS_CYCLES + busy) / sweeps;
}

static double search(const Fields& fields, int sms)
{
    double least = 1e300, points = 0;
    const int most_side = 148;
    for (const auto& f : fields) points += (double)(f.first - 2) * (f.second - 2);
    const int fewest = std::max(1, (int)std::ceil(points / ((double)sms * most_side * most_side)));
    for (int per_sm = fewest; per_sm < fewest + 3; ++per_sm)
        for (double factor = 0.94; factor < 1.6; factor *= 1.02)
            for (double flat : {1.0, 0.87, 0.75}) {
                const int sx = (int)std::min<double>(most_side, std::max(6.0, std::sqrt(points / ((double)sms * per_sm)) * factor));
                const int sy = (int)std::max(6.0, sx * flat);
                // the fields' sums once a pair, as the search had them
                for (int sweeps = 1; sweeps <= 6; ++sweeps) {
                    const double c = cost_of(fields, sms, sweeps, sx, sy);
                    if (c < least) least = c;
                }
            }
    return least;
}

int main()
{
    std::mt19937 rng(3);
    auto sides = [&](int lo, int hi) { return lo + (int)(rng() % (unsigned)(hi - lo + 1)); };
    double worst = 0;
    for (int k = 0; k < 300; ++k) {
        Fields f;
        const int count = 1 + (int)(rng() % (k % 3 == 0 ? 4 : k % 3 == 1 ? 40 : 300));
        const int lo = 3 << (rng() % 6), hi = lo + 1 + (int)(rng() % 900);
        for (int c = 0; c < count; ++c) {
            if (c > 0 && rng() % 3 == 0) f.push_back(f[rng() % f.size()]);
            else f.push_back({sides(lo, hi), sides(lo, hi)});
        }
        const BatchSweepPlan p = plan_batch_sweeps(f, 152);
        if (p.sweeps < 1 || p.sx < 1 || p.sy < 1) return 1;
        worst = std::max(worst, cost_of(f, 152, p.sweeps, p.sx, p.sy) / search(f, 152));
    }
    Fields many;
    for (int c = 0; c < 1000; ++c) many.push_back({sides(33, 97), sides(33, 97)});
    auto least_time = [&](auto&& run) {
        double t = 1e300;
        for (int k = 0; k < 25; ++k) {
            const auto a = std::chrono::steady_clock::now();
            run();
            t = std::min(t, std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - a).count());
        }
        return t;
    };
    volatile double sink = 0;
    const double fast = least_time([&] { sink = sink + plan_batch_sweeps(many, 152).sweeps; });
    // one evaluation of every pair (the search above takes six, one for each number of sweeps)
    const double plain = least_time([&] {
        for (int k = 0; k < 243; ++k) sink = sink + cost_of(many, 152, 1 + k % 6, 40 + k % 30, 40 + k % 30);
    });
    std::printf("%.6f %.1f %.1f\n", worst, fast, plain);
    return 0;
}
