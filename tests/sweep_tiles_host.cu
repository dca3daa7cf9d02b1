// Host side of sweep_tiles.cu without a GPU: its launches are recorded instead of made. Reads "m n sms" lines
// and checks that the dynamic shared memory of every launch that a plan leads to holds the windows of its
// tiles, and no more than a CTA can have. Prints the launches looked at, the failures and how many plans have
// one sweep to a launch (those lead to launches of none: an even number of launches is made).
#include <cuda_runtime.h>

#include <cstdio>

static size_t g_bytes;
template <class... P, class... A>
cudaError_t record_launch(const cudaLaunchConfig_t* c, void (*)(P...), A...)
{
    g_bytes = c->dynamicSmemBytes;
    return cudaSuccess;
}
#define cudaLaunchKernelEx record_launch
#define cudaGetLastError() cudaSuccess
#include "sweep_tiles.cu"

namespace lap {
void note_launch() {}
}  // namespace lap
using namespace lap;

// Bytes of the largest window of the launch's tiles, as the kernel cuts them.
static int64_t window_bytes(int m, int n, const SweepTiles& t, int kind, int sweeps)
{
    const int h = std::max(1, kind == SWEEP_JACOBI ? sweeps : 2 * sweeps);
    int64_t worst = 0;
    for (int bx = 0; bx < t.tx; ++bx)
        for (int by = 0; by < t.ty; ++by) {
            const int x0 = 1 + (int)((int64_t)bx * (m - 2) / t.tx), x1 = 1 + (int)((int64_t)(bx + 1) * (m - 2) / t.tx);
            const int y0 = 1 + (int)((int64_t)by * (n - 2) / t.ty), y1 = 1 + (int)((int64_t)(by + 1) * (n - 2) / t.ty);
            const int64_t W = std::min(m, x1 + h) - std::max(0, x0 - h), H = std::min(n, y1 + h) - std::max(0, y0 - h);
            worst = std::max(worst, W * H * 8 * (kind == SWEEP_JACOBI ? 2 : 1));
        }
    return worst;
}

int main()
{
    long long launches = 0, bad = 0, single = 0;
    int m, n, sms;
    while (std::scanf("%d %d %d", &m, &n, &sms) == 3)
        for (int kind : {SWEEP_JACOBI, SWEEP_SOR, SWEEP_GS})
            for (int form = 0; form < 4; ++form) {  // 1/d a power of two with beta = 1 or not, no power, diagonal pairs
                const bool diag = form == 3;
                if (diag && kind == SWEEP_JACOBI) continue;
                Coef c{};
                c.b2 = form == 1 ? 3.0 : form == 2 ? 0.64 : 1.0;
                c.d = 2.0 * (1.0 + c.b2);
                c.inv_d = 1.0 / c.d;
                c.unit_beta = c.b2 == 1.0;
                c.inv_d_shift = form == 1 ? 3 : form == 2 ? 0 : 2;
                const SweepTiles t = plan_sweep_tiles(m, n, c, kind, diag, sms);
                if (!t.sweeps) continue;
                single += t.sweeps == 1;
                for (int s = t.sweeps == 1 ? 0 : 1; s <= t.sweeps; ++s) {
                    launch_sweep_tiles(Field{nullptr, m, n, m}, nullptr, m, c, t, kind, diag, s, true, nullptr, nullptr);
                    const int64_t need = window_bytes(m, n, t, kind, s);
                    ++launches;
                    if ((int64_t)g_bytes >= need && g_bytes <= 227 * 1024) continue;
                    if (++bad <= 5)
                        std::fprintf(stderr, "%d x %d, kind %d form %d: a launch of %d sweeps has %zu bytes, needs %lld\n", m, n,
                                     kind, form, s, g_bytes, (long long)need);
                }
            }
    std::printf("%lld %lld %lld\n", launches, bad, single);
    return 0;
}
