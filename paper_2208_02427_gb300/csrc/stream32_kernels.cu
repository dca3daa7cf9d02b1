// stream32_kernels.cu -- the FP32 V-cycle's work on a level as streams of rows through registers.
//
// A level's whole descent (nu smoothing sweeps from a zero correction, the residual, full
// weighting) and its whole ascent (interpolation, nu sweeps, and on level 0 the FP64 update
// psi += e) are one pass over memory each. A warp takes a block of up to 128 columns, four
// consecutive ones per lane, and runs down a strip of rows. Every step loads one row and advances
// each colour pass by one row: with row y loaded, pass p (p = 0, 1, 2, ...: red, black, red, ...)
// updates row y - p, whose neighbours are up to date. The rows in flight live in registers, west
// and east neighbours come by shuffle, and no step waits for another warp: there is no shared
// tile, no barrier and no second look at a value. Halo rows and columns are recomputed by the
// neighbouring warps; blocks at the domain's edge need none, as the ring is zero.
//
// What bounds it: memory on levels above the L2's size, and the number of row steps times a
// step's dependent chain on small ones. The shared-memory tiles this replaces were bound by
// shared-memory traffic and barriers (issue slots 45-59% busy).
//
// Every value is the per-pass kernels' value bit for bit (same expressions, same rounding): E and
// O hold a row's even and odd columns, and since a pass p is one row behind pass p - 1 and of the
// other colour, all passes of a step update the same one of the two, E on even steps and O on odd
// ones. Points of the ring and outside are kept at zero by a zero in place of 1/d.
#include <algorithm>
#include <type_traits>

#include "lap_device.cuh"
#include "lap_internal.cuh"

namespace lap {

namespace {

constexpr unsigned ALL = 0xffffffffu;
constexpr int ST_WARPS = 4;  // warps per CTA
constexpr int STREAM_WARPS_PER_SM = 16;

// Row pipelines are unrolled over their D rows in flight in registers; rows come from memory R
// ahead (R divides D, so that a row's slot is known at compile time).
__host__ __device__ constexpr int depth_of(int nu) { return 2 * nu + 2; }
__host__ __device__ constexpr int ahead(int depth) { return depth <= 6 ? depth : depth / 2; }
// floats of shared memory per warp: the rings of q (descent), of q, u, psi (double) and of coarse
// rows (64 values and one beyond each segment's last lane, D / 2 rows; ascent)
__host__ __device__ constexpr int down_ring(int nu) { return 128 * ahead(depth_of(nu)); }
constexpr int COARSE_ROW = 72;
__host__ __device__ constexpr int up_ring(int nu, bool psi)
{
    return 128 * ahead(depth_of(nu)) * (psi ? 4 : 2) + COARSE_ROW * (depth_of(nu) / 2);
}

struct Pair {  // columns c0, c2 (e) and c1, c3 (o) of a lane's four
    float2 e, o;
};

struct StreamCoef {
    float2 b2, d, w, omw;
    float2 inv_e, inv_o;  // 1/d per column, 0 on the ring and outside
};

__device__ __forceinline__ float2 pair2(float v) { return make_float2(v, v); }

// f v, for a product that is added next: the compiler joins a packed product and a packed sum to
// one multiply-add (also under --fmad=false), which halves and quarters show below FP32's normal
// range, where they round. Scalar products stay separate.
__device__ __forceinline__ float2 times2(float f, float2 v)
{
    return make_float2(__fmul_rn(f, v.x), __fmul_rn(f, v.y));
}

__device__ __forceinline__ void cp16(unsigned dst, const void* src, int bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
template <int B>
__device__ __forceinline__ void cp_small(unsigned dst, const void* src, int bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(dst), "l"(src), "n"(B), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// West and east neighbours of the E points (from O) or of the O points (from E) of row c. sw: lanes
// per segment; past a segment's last lane lies the ring or a halo column that nothing uses.
template <bool E>
__device__ __forceinline__ void west_east(const Pair& c, int sw, bool last, float2& w, float2& e)
{
    if (E) {
        const float l = __shfl_up_sync(ALL, c.o.y, 1, sw);
        w = make_float2(l, c.o.x);
        e = c.o;
    } else {
        float r = __shfl_down_sync(ALL, c.e.x, 1, sw);
        r = last ? 0.f : r;
        w = c.e;
        e = make_float2(c.e.y, r);
    }
}

// (E + W) + b2 (N + S) + q of the E or O points of row c with rows s below and n above.
template <bool E, bool UNIT>
__device__ __forceinline__ float2 stencil(const Pair& c, const Pair& s, const Pair& n, const Pair& q,
                                          const StreamCoef& k, int sw, bool last)
{
    float2 w, e;
    west_east<E>(c, sw, last, w, e);
    const float2 ew = __fadd2_rn(w, e);
    const float2 ns = __fadd2_rn(E ? s.e : s.o, E ? n.e : n.o);
    const float2 t = UNIT ? __fadd2_rn(ns, ew) : __ffma2_rn(k.b2, ns, ew);
    return __fadd2_rn(t, E ? q.e : q.o);
}

// Eq. 6 (GS) or Eq. 7 on the E or O points of row c; in: whether the row is an interior one.
template <bool E, bool UNIT, bool GS>
__device__ __forceinline__ void relax(Pair& c, const Pair& s, const Pair& n, const Pair& q,
                                      const StreamCoef& k, int sw, bool last, bool in)
{
    const float2 t = stencil<E, UNIT>(c, s, n, q, k, sw, last);
    float2 iv = E ? k.inv_e : k.inv_o;
    iv.x = in ? iv.x : 0.f;
    iv.y = in ? iv.y : 0.f;
    float2 g = __fmul2_rn(t, iv);
    float2& v = E ? c.e : c.o;
    if (!GS) g = __ffma2_rn(k.w, g, __fmul2_rn(k.omw, v));
    v = g;
}

// What a lane works on.
struct Lane {
    int col;       // its first column (a multiple of 4)
    int sw;        // lanes per segment
    bool last;     // the segment's last lane
    bool owner;    // its columns are stored by this warp
    int y0, y1;    // rows stored by this segment
};

__device__ __forceinline__ Lane lane_of(const StreamItem& it, int n)
{
    Lane a;
    const int lane = threadIdx.x & 31;
    a.sw = 1 << it.sw_log;
    const int l = lane & (a.sw - 1), seg = lane >> it.sw_log;
    a.col = it.gx0 + 4 * l;
    a.last = l == a.sw - 1;
    a.owner = a.col >= it.x0 && a.col < it.x1;
    a.y0 = it.y0 + seg * it.rows;
    a.y1 = min(a.y0 + it.rows, n);
    return a;
}

__device__ __forceinline__ StreamCoef coefs(const BatchLevel<float>& F, int col, float w, float omw)
{
    StreamCoef k;
    k.b2 = pair2((float)F.b2);
    k.d = pair2(-(float)F.d);
    k.w = pair2(w);
    k.omw = pair2(omw);
    const float iv = (float)F.inv_d;
    auto inside = [&](int c) { return c >= 1 && c <= F.m - 2 ? iv : 0.f; };
    k.inv_e = make_float2(inside(col), inside(col + 2));
    k.inv_o = make_float2(inside(col + 1), inside(col + 3));
    return k;
}

// Rows of an array in flight from memory: a ring of rows per warp in shared memory, 16 bytes a
// lane, each lane reading back what it fetched. Rows outside [0, n) and columns outside [0, m) are
// zero.
struct RowRing {
    unsigned slot;  // shared address of this lane's 16 bytes in slot 0
    const float *src, *base;
    int64_t pitch;
    int bytes, n;
    __device__ __forceinline__ RowRing(float* smem, const float* src, int64_t p, int col, int m, int rows)
        : slot((unsigned)__cvta_generic_to_shared(smem + 4 * (threadIdx.x & 31))), src(src), base(src + col),
          pitch(p), bytes(col < 0 ? 0 : max(0, min(16, 4 * (m - col)))), n(rows)
    {
    }
    __device__ __forceinline__ void fetch(int k, int y, bool on = true) const
    {
        const bool in = on && y >= 0 && y < n && bytes > 0;
        cp16(slot + 512 * k, in ? base + (int64_t)y * pitch : src, in ? bytes : 0);
    }
    __device__ __forceinline__ Pair take(int k) const
    {
        float4 v;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                     : "r"(slot + 512 * k));
        return Pair{make_float2(v.x, v.z), make_float2(v.y, v.w)};
    }
};

// ---- descent ------------------------------------------------------------------------------
// NU sweeps on level F from u = 0 with source q, the residual, and the restricted residual of the
// coarse points whose centre the segment owns to C.q, the smoothed u to F.r; zero_c: C.u := 0.
template <int NU, bool UNIT, bool GS>
__device__ __forceinline__ void stream_down(const StreamItem& it, const BatchLevel<float>& F,
                                            const BatchLevel<float>& C, float w, float omw, bool zero_c,
                                            float* smem)
{
    constexpr int D = depth_of(NU), R = ahead(D);
    const int m = F.m, n = F.n;
    const Lane a = lane_of(it, n);
    const StreamCoef k = coefs(F, a.col, w, omw);
    const RowRing ring(smem, F.q, F.pitch, a.col, m, n);
    // rows y0 - D .. y1 - 1 + 2 NU are loaded; a warp runs the steps of its tallest segment
    const int ybase = a.y0 - D;
    const int steps = it.rows + 4 * NU + 2;
    const bool work = a.y0 < a.y1;
    Pair U[D], Q[D];
#pragma unroll
    for (int s = 0; s < D; ++s) U[s].e = U[s].o = Q[s].e = Q[s].o = pair2(0.f);
#pragma unroll
    for (int s = 0; s < R; ++s) {
        ring.fetch(s, ybase + s, work);
        cp_commit();
    }
    const int mc = (m - 1) / 2 + 1, nc = (n - 1) / 2 + 1;
    const int I = a.col >> 1;  // the coarse columns of this lane: I, I + 1
    const bool own0 = a.owner && I >= 1 && I <= mc - 2, own1 = a.owner && I + 1 <= mc - 2;
    float2 south = pair2(0.f), sx = pair2(0.f), centre = pair2(0.f), we = pair2(0.f);
    for (int t = 0; t < steps; t += D) {
#pragma unroll
        for (int K = 0; K < D; ++K) {
            const int y = ybase + t + K;
            cp_wait<R - 1>();
            Q[K] = ring.take(K % R);
            // pass 0 (red) on row y: the neighbours are zero, s = 0 + q
            const bool in0 = y >= 1 && y <= n - 2;
            if ((K & 1) == 0) {
                float2 iv = make_float2(in0 ? k.inv_e.x : 0.f, in0 ? k.inv_e.y : 0.f);
                float2 g = __fmul2_rn(__fadd2_rn(pair2(0.f), Q[K].e), iv);
                if (!GS) g = __ffma2_rn(k.w, g, __fmul2_rn(k.omw, pair2(0.f)));
                U[K].e = g;
                U[K].o = pair2(0.f);
            } else {
                float2 iv = make_float2(in0 ? k.inv_o.x : 0.f, in0 ? k.inv_o.y : 0.f);
                float2 g = __fmul2_rn(__fadd2_rn(pair2(0.f), Q[K].o), iv);
                if (!GS) g = __ffma2_rn(k.w, g, __fmul2_rn(k.omw, pair2(0.f)));
                U[K].o = g;
                U[K].e = pair2(0.f);
            }
            // passes 1 .. 2 NU - 1 on rows y - 1 .. y - 2 NU + 1
#pragma unroll
            for (int p = 1; p < 2 * NU; ++p) {
                const int r = y - p;
                const bool in = r >= 1 && r <= n - 2;
                Pair& c = U[(K - p + D) % D];
                const Pair &s = U[(K - p - 1 + D) % D], &nn = U[(K - p + 1 + D) % D], &q = Q[(K - p + D) % D];
                if ((K & 1) == 0) relax<true, UNIT, GS>(c, s, nn, q, k, a.sw, a.last, in);
                else relax<false, UNIT, GS>(c, s, nn, q, k, a.sw, a.last, in);
            }
            {  // row y - 2 NU + 1 is final
                const int r = y - 2 * NU + 1;
                const Pair& c = U[(K - 2 * NU + 1 + D) % D];
                if (a.owner && a.col < m && r >= max(1, a.y0) && r < min(a.y1, n - 1))
                    *reinterpret_cast<float4*>(F.r + (int64_t)r * F.pitch + a.col) =
                        make_float4(c.e.x, c.o.x, c.e.y, c.o.y);
            }
            // the residual of row r = y - 2 NU, E and O points
            const int r = y - 2 * NU;
            const Pair &c = U[(K - 2 * NU + D) % D], &s = U[(K - 2 * NU - 1 + D) % D],
                       &nn = U[(K - 2 * NU + 1 + D) % D], &q = Q[(K - 2 * NU + D) % D];
            const float2 re = __ffma2_rn(k.d, c.e, stencil<true, UNIT>(c, s, nn, q, k, a.sw, a.last));
            const float2 ro = __ffma2_rn(k.d, c.o, stencil<false, UNIT>(c, s, nn, q, k, a.sw, a.last));
            const float rl = __shfl_up_sync(ALL, ro.y, 1, a.sw);
            const float2 x = __fadd2_rn(make_float2(rl, ro.x), ro);  // odd columns left + right
            if ((K & 1) == 0) {  // an even row: centres, west + east
                centre = re;
                we = x;
            } else {  // an odd row: north of coarse row (r - 1) / 2, south of the next
                const int J = (r - 1) >> 1;
                const float2 edges = __fadd2_rn(we, __fadd2_rn(south, re));
                const float2 corners = __fadd2_rn(sx, x);
                const float2 tt = __ffma2_rn(pair2(2.f), centre, edges);
                const float2 v = __fmul2_rn(pair2(0.25f), __ffma2_rn(pair2(2.f), tt, corners));
                if (J >= 1 && J <= nc - 2 && 2 * J >= a.y0 && 2 * J < a.y1) {
                    const int64_t at = (int64_t)J * C.pitch + I;
                    if (own0 && own1) {
                        *reinterpret_cast<float2*>(C.q + at) = v;
                        if (zero_c) *reinterpret_cast<float2*>(C.u + at) = pair2(0.f);
                    } else if (own0) {
                        C.q[at] = v.x;
                        if (zero_c) C.u[at] = 0.f;
                    } else if (own1) {
                        C.q[at + 1] = v.y;
                        if (zero_c) C.u[at + 1] = 0.f;
                    }
                }
                south = re;
                sx = x;
            }
            ring.fetch(K % R, y + R, work);
            cp_commit();
        }
    }
    cp_wait<0>();
}

// ---- ascent -------------------------------------------------------------------------------
// u (the descent's, in F.r) plus the bilinear interpolation of C.u, then NU sweeps; the result to
// F.u, or added to the FP64 field psi (level 0 of the mixed solver's last inner cycle). The
// interpolation works on row y, pass p on row y - 1 - p. With Gauss-Seidel the red points' values
// before the first red pass are never read, so only the black points are interpolated.
// (Computing the descent's sweeps again from q in front of this pipeline, instead of storing u in
// the descent and reading it here, saves a quarter of the bytes; but the longer pipeline spilled at
// 168 registers: 8193^2 with the update 551 us against 359 us, plus 30 us less in the descent.)
template <int NU, bool UNIT, bool GS, bool PSI>
__device__ __forceinline__ void stream_up(const StreamItem& it, const BatchLevel<float>& F,
                                          const BatchLevel<float>& C, float w, float omw, double* psi,
                                          int64_t psi_pitch, float* smem)
{
    constexpr int D = depth_of(NU), R = ahead(D);
    constexpr int LAST = 2 * NU;  // row y - LAST is final
    const int m = F.m, n = F.n;
    const Lane a = lane_of(it, n);
    const StreamCoef k = coefs(F, a.col, w, omw);
    const RowRing qring(smem, F.q, F.pitch, a.col, m, n);
    const RowRing uring(smem + 128 * R, F.r, F.pitch, a.col, m, n);
    const int ybase = a.y0 - LAST;
    const int steps = it.rows + 2 * LAST;
    const bool work = a.y0 < a.y1;
    // psi rows: 32 bytes a lane, in two halves of 16 (this lane's columns c0, c1 and c2, c3)
    unsigned pslot = 0;
    int pb0 = 0, pb1 = 0;
    bool vec = false;
    if (PSI) {
        pslot = (unsigned)__cvta_generic_to_shared(smem + 128 * R * 2 + 8 * (threadIdx.x & 31));
        vec = (reinterpret_cast<uintptr_t>(psi) & 15) == 0 && (psi_pitch & 1) == 0;
        pb0 = a.owner && vec ? max(0, min(16, 8 * (m - a.col))) : 0;
        pb1 = a.owner && vec ? max(0, min(16, 8 * (m - a.col - 2))) : 0;
    }
    auto psi_fetch = [&](int slot, int r) {
        const bool in = work && r >= max(1, a.y0) && r < min(a.y1, n - 1);
        const double* p = psi + (in ? (int64_t)r * psi_pitch + a.col : 0);
        const unsigned s = pslot + 1024 * slot;
        if (in && pb0 > 0) cp16(s, p, pb0);
        if (in && pb1 > 0) cp16(s + 16, p + 2, pb1);
    };
    // Coarse rows: cur = row floor(y / 2), nxt the one above. An odd step takes the next one from a
    // ring of D / 2 rows, a slot per odd step of the unrolled D.
    constexpr int RC = D / 2;
    const int mc = (m - 1) / 2 + 1, nc = (n - 1) / 2 + 1, I = a.col >> 1;
    struct Coarse {
        float2 v;
        float right;  // the value beyond a segment's last lane
    };
    const int lane = threadIdx.x & 31;
    const unsigned cslot = (unsigned)__cvta_generic_to_shared(smem + 128 * R * (PSI ? 4 : 2) + 2 * lane);
    const unsigned rslot = cslot + 4 * (64 - 2 * lane + (lane >> it.sw_log));
    const int cbytes = a.col < 0 ? 0 : max(0, min(8, 4 * (mc - I))), rbytes = a.last && I + 2 < mc && a.col >= 0 ? 4 : 0;
    const float* cbase = C.u + (cbytes > 0 ? I : 0);
    auto coarse_fetch = [&](int slot, int J) {
        const bool in = work && J >= 0 && J < nc;
        const float* p = cbase + (in ? (int64_t)J * C.pitch : 0);
        cp_small<8>(cslot + 4 * COARSE_ROW * slot, p, in ? cbytes : 0);
        if (a.last) cp_small<4>(rslot + 4 * COARSE_ROW * slot, rbytes > 0 ? p + 2 : p, in ? rbytes : 0);
    };
    auto coarse_take = [&](int slot) {
        Coarse c{pair2(0.f), 0.f};
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(c.v.x), "=f"(c.v.y) : "r"(cslot + 4 * COARSE_ROW * slot));
        if (a.last) asm volatile("ld.shared.f32 %0, [%1];" : "=f"(c.right) : "r"(rslot + 4 * COARSE_ROW * slot));
        return c;
    };
    const int J0 = ybase >> 1;  // ybase is even
#pragma unroll
    for (int i = 0; i < RC; ++i) coarse_fetch(i, J0 + 1 + i);
    Coarse cur{pair2(0.f), 0.f}, nxt{pair2(0.f), 0.f};
    if (work && J0 >= 0 && J0 < nc && cbytes > 0) {
        const float* p = cbase + (int64_t)J0 * C.pitch;
        cur.v.x = p[0];
        if (cbytes > 4) cur.v.y = p[1];
        if (rbytes > 0) cur.right = p[2];
    }
    Pair U[D], Q[D];
#pragma unroll
    for (int s = 0; s < D; ++s) U[s].e = U[s].o = Q[s].e = Q[s].o = pair2(0.f);
#pragma unroll
    for (int s = 0; s < R; ++s) {
        qring.fetch(s, ybase + s, work);
        uring.fetch(s, ybase + s, work);
        cp_commit();
    }
    const FmaOps o = load_fma_ops();
    for (int t = 0; t < steps; t += D) {
#pragma unroll
        for (int K = 0; K < D; ++K) {
            const int y = ybase + t + K;
            cp_wait<R - 1>();
            Q[K] = qring.take(K % R);
            U[K] = uring.take(K % R);
            // interpolation on row y: even rows take coarse row y / 2, odd rows the mean
            // of it and the next; even columns one coarse column, odd columns the mean of two.
            // Black points: odd columns of even rows, even columns of odd rows.
            {
                const bool in = y >= 1 && y <= n - 2;
                Pair& c = U[K];
                float2 pe = pair2(0.f), po = pair2(0.f);
                if (K & 1) nxt = coarse_take(K / 2);
                if ((K & 1) == 0) {
                    float rt = __shfl_down_sync(ALL, cur.v.x, 1, a.sw);
                    rt = a.last ? cur.right : rt;
                    if (!GS) pe = cur.v;
                    po = times2(0.5f, __fadd2_rn(cur.v, make_float2(cur.v.y, rt)));
                } else {
                    pe = times2(0.5f, __fadd2_rn(cur.v, nxt.v));
                    if (!GS) {
                        float r0 = __shfl_down_sync(ALL, cur.v.x, 1, a.sw);
                        float r1 = __shfl_down_sync(ALL, nxt.v.x, 1, a.sw);
                        r0 = a.last ? cur.right : r0;
                        r1 = a.last ? nxt.right : r1;
                        po = times2(0.25f, __fadd2_rn(__fadd2_rn(cur.v, make_float2(cur.v.y, r0)),
                                                      __fadd2_rn(nxt.v, make_float2(nxt.v.y, r1))));
                    }
                }
                // the ring and the columns outside stay as they are (a zero 1/d marks them)
                const bool eo = !GS || (K & 1), oo = !GS || (K & 1) == 0;
                if (eo) {
                    const float2 v = __fadd2_rn(c.e, pe);
                    if (in && k.inv_e.x != 0.f) c.e.x = v.x;
                    if (in && k.inv_e.y != 0.f) c.e.y = v.y;
                }
                if (oo) {
                    const float2 v = __fadd2_rn(c.o, po);
                    if (in && k.inv_o.x != 0.f) c.o.x = v.x;
                    if (in && k.inv_o.y != 0.f) c.o.y = v.y;
                }
                if (K & 1) {
                    cur = nxt;
                    coarse_fetch(K / 2, ((y + 1) >> 1) + RC);
                }
            }
            // passes 0 .. 2 NU - 1 on rows y - 1, y - 2, ..: O points on even steps, E on odd ones
#pragma unroll
            for (int p = 0; p < 2 * NU; ++p) {
                const int r = y - 1 - p;
                const bool in = r >= 1 && r <= n - 2;
                Pair& c = U[(K - 1 - p + D) % D];
                const Pair &s = U[(K - 2 - p + D) % D], &nn = U[(K - p + D) % D], &q = Q[(K - 1 - p + D) % D];
                if (K & 1) relax<true, UNIT, GS>(c, s, nn, q, k, a.sw, a.last, in);
                else relax<false, UNIT, GS>(c, s, nn, q, k, a.sw, a.last, in);
            }
            // row r = y - LAST is final
            const int r = y - LAST;
            const Pair& c = U[(K - LAST + D) % D];
            const bool mine = work && a.owner && a.col < m && r >= max(1, a.y0) && r < min(a.y1, n - 1);
            if (!PSI) {
                if (mine)
                    *reinterpret_cast<float4*>(F.u + (int64_t)r * F.pitch + a.col) =
                        make_float4(c.e.x, c.o.x, c.e.y, c.o.y);
            } else {
                if (mine) {
                    double* p = psi + (int64_t)r * psi_pitch + a.col;
                    const bool i0 = k.inv_e.x != 0.f, i1 = k.inv_o.x != 0.f, i2 = k.inv_e.y != 0.f,
                               i3 = k.inv_o.y != 0.f;
                    double v0, v1, v2, v3;
                    if (vec) {
                        const unsigned s = pslot + 1024 * (K % R);
                        asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v0), "=d"(v1) : "r"(s));
                        asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v2), "=d"(v3) : "r"(s + 16));
                    } else {
                        v0 = i0 ? p[0] : 0.0;
                        v1 = i1 ? p[1] : 0.0;
                        v2 = i2 ? p[2] : 0.0;
                        v3 = i3 ? p[3] : 0.0;
                    }
                    v0 = fadd(o, v0, to_double_exact(c.e.x));
                    v1 = fadd(o, v1, to_double_exact(c.o.x));
                    v2 = fadd(o, v2, to_double_exact(c.e.y));
                    v3 = fadd(o, v3, to_double_exact(c.o.y));
                    if (vec && i0 && i1) {
                        *reinterpret_cast<double2*>(p) = make_double2(v0, v1);
                    } else {
                        if (i0) p[0] = v0;
                        if (i1) p[1] = v1;
                    }
                    if (vec && i2 && i3) {
                        *reinterpret_cast<double2*>(p + 2) = make_double2(v2, v3);
                    } else {
                        if (i2) p[2] = v2;
                        if (i3) p[3] = v3;
                    }
                }
            }
            qring.fetch(K % R, y + R, work);
            uring.fetch(K % R, y + R, work);
            if (PSI) psi_fetch(K % R, r + R);
            cp_commit();
        }
    }
    cp_wait<0>();
}

// ---- kernels --------------------------------------------------------------------------------
// Warp `index` of the launch: an item of the list, or (no list) the index-th piece of level
// `level` cut as StreamCut says.
__device__ __forceinline__ bool stream_item(const StreamItem* items, int count, const StreamCut& cut,
                                            int index, StreamItem* it)
{
    if (index >= count) return false;
    if (items) *it = items[index];
    else *it = stream_piece(cut, index);
    return true;
}

// CTAs per SM: four at 128 registers a thread where the pipeline fits them, else three at 168.
__host__ __device__ constexpr int down_ctas(int nu, bool gs) { return nu == 3 || (nu == 2 && !gs) ? 3 : 4; }
__host__ __device__ constexpr int up_ctas(int nu, bool gs, bool psi)
{
    return nu == 3 || (nu == 2 && !gs) || (nu == 2 && psi) ? 3 : 4;
}

template <int NU, bool GS>
__global__ void __launch_bounds__(32 * ST_WARPS, down_ctas(NU, GS))
    stream_down_kernel(const StreamItem* __restrict__ items, int count, StreamCut cut,
                       const BatchLevel<float>* __restrict__ lv, const int* __restrict__ active, float w,
                       float omw, int zero_c)
{
    after_prior();
    extern __shared__ float4 smem4[];
    const int wid = threadIdx.x >> 5;
    float* smem = reinterpret_cast<float*>(smem4) + wid * down_ring(NU);
    StreamItem it;
    if (!stream_item(items, count, cut, blockIdx.x * ST_WARPS + wid, &it)) return;
    const BatchLevel<float> F = lv[it.level];
    if (active && !active[F.problem]) return;
    const BatchLevel<float> C = lv[it.level + 1];
    if (F.unit_beta) stream_down<NU, true, GS>(it, F, C, w, omw, zero_c != 0, smem);
    else stream_down<NU, false, GS>(it, F, C, w, omw, zero_c != 0, smem);
}

template <int NU, bool GS, bool PSI>
__global__ void __launch_bounds__(32 * ST_WARPS, up_ctas(NU, GS, PSI))
    stream_up_kernel(const StreamItem* __restrict__ items, int count, StreamCut cut,
                     const BatchLevel<float>* __restrict__ lv, const int* __restrict__ active, float w,
                     float omw, double* psi, int64_t psi_pitch, const BatchLevel<double>* __restrict__ lv64)
{
    after_prior();
    extern __shared__ float4 smem4[];
    const int wid = threadIdx.x >> 5;
    float* smem = reinterpret_cast<float*>(smem4) + wid * up_ring(NU, PSI);
    StreamItem it;
    if (!stream_item(items, count, cut, blockIdx.x * ST_WARPS + wid, &it)) return;
    const BatchLevel<float> F = lv[it.level];
    if (active && !active[F.problem]) return;
    const BatchLevel<float> C = lv[it.level + 1];
    if (PSI && lv64) {
        psi = lv64[it.level].u;
        psi_pitch = lv64[it.level].pitch;
    }
    if (F.unit_beta) stream_up<NU, true, GS, PSI>(it, F, C, w, omw, psi, psi_pitch, smem);
    else stream_up<NU, false, GS, PSI>(it, F, C, w, omw, psi, psi_pitch, smem);
}

int round_up4(int v) { return (v + 3) / 4 * 4; }

// The cut of a level for a pipeline of D rows that needs `extra` steps beyond a strip's rows and
// halo columns hl, hr, into about `warps` pieces (at most, unless strips get shorter than 8 rows).
StreamCut cut_level(int level, int m, int n, int D, int extra, int hl, int hr, int64_t warps)
{
    StreamCut c;
    c.level = level;
    c.m = m;
    c.n = n;
    c.hl = hl;
    c.hr = hr;
    c.sw_log = m - 1 <= 16 ? 2 : (m - 1 <= 32 ? 3 : (m - 1 <= 64 ? 4 : 5));
    const int width = 4 << c.sw_log, segs = 32 >> c.sw_log;
    c.nb = 1;
    if (m - 1 > width)
        for (int x = width - hr;; x += width - hl - hr) {
            ++c.nb;
            if (m - 1 - (x - hl) <= width) break;
        }
    // rows: even, rows + extra a multiple of D; rows 0 .. n - 2 have something to store
    int rows = 8;
    while ((rows + extra) % D != 0 || (rows & 1)) ++rows;
    auto strips = [&](int r) { return (n - 1 + r * segs - 1) / (r * segs); };
    while ((int64_t)c.nb * strips(rows) > warps && rows < n) rows += D;
    c.rows = rows;
    c.strips = strips(rows);
    return c;
}

StreamCut down_cut(int level, int m, int n, int nu, int64_t warps)
{
    return cut_level(level, m, n, depth_of(nu), 4 * nu + 2, round_up4(2 * nu + 1), round_up4(2 * nu), warps);
}

StreamCut up_cut(int level, int m, int n, int nu, int64_t warps)
{
    return cut_level(level, m, n, depth_of(nu), 4 * nu, round_up4(2 * nu), round_up4(2 * nu), warps);
}

template <int NU, bool GS>
cudaError_t down_launch(const StreamItem* items, int count, const StreamCut& cut, const BatchLevel<float>* lv,
                        const int* active, float w, float omw, bool zero_c, cudaStream_t s)
{
    launch_after(stream_down_kernel<NU, GS>, (count + ST_WARPS - 1) / ST_WARPS, 32 * ST_WARPS, ST_WARPS * down_ring(NU) * sizeof(float), s, items, count, cut, lv, active, w,
                                                                                omw, zero_c ? 1 : 0);
    note_launch();
    return cudaGetLastError();
}

template <int NU, bool GS, bool PSI>
cudaError_t up_launch(const StreamItem* items, int count, const StreamCut& cut, const BatchLevel<float>* lv,
                      const int* active, float w, float omw, double* psi, int64_t psi_pitch,
                      const BatchLevel<double>* lv64, cudaStream_t s)
{
    auto kern = stream_up_kernel<NU, GS, PSI>;
    const size_t smem = ST_WARPS * up_ring(NU, PSI) * sizeof(float);
    static std::atomic<size_t> set[ATTR_DEVICES];
    const int dev = attr_slot();
    if (smem > 48 * 1024 && !(dev >= 0 && set[dev].load() >= smem)) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr_record(set, dev, smem);
    }
    launch_after(kern, (count + ST_WARPS - 1) / ST_WARPS, 32 * ST_WARPS, smem, s, items, count, cut, lv, active, w, omw, psi,
                                                                         psi_pitch, lv64);
    note_launch();
    return cudaGetLastError();
}

template <class F>
cudaError_t on_nu(int nu, F&& f)
{
    switch (nu) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 3: return f(std::integral_constant<int, 3>{});
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t down(const StreamItem* items, int count, const StreamCut& cut, const BatchLevel<float>* lv,
                 const int* active, int nu, bool gs, double w, bool zero_c, cudaStream_t s)
{
    const float wf = (float)w, omw = (float)(1.0 - w);
    return on_nu(nu, [&](auto N) {
        return gs ? down_launch<N.value, true>(items, count, cut, lv, active, wf, omw, zero_c, s)
                  : down_launch<N.value, false>(items, count, cut, lv, active, wf, omw, zero_c, s);
    });
}

cudaError_t up(const StreamItem* items, int count, const StreamCut& cut, const BatchLevel<float>* lv,
               const int* active, int nu, bool gs, double w, double* psi, int64_t psi_pitch,
               const BatchLevel<double>* lv64, cudaStream_t s)
{
    const float wf = (float)w, omw = (float)(1.0 - w);
    const bool fold = psi != nullptr || lv64 != nullptr;
    return on_nu(nu, [&](auto N) {
        if (gs)
            return fold ? up_launch<N.value, true, true>(items, count, cut, lv, active, wf, omw, psi, psi_pitch, lv64, s)
                        : up_launch<N.value, true, false>(items, count, cut, lv, active, wf, omw, psi, psi_pitch, lv64, s);
        return fold ? up_launch<N.value, false, true>(items, count, cut, lv, active, wf, omw, psi, psi_pitch, lv64, s)
                    : up_launch<N.value, false, false>(items, count, cut, lv, active, wf, omw, psi, psi_pitch, lv64, s);
    });
}

// Warps a single grid's level is cut into.
int64_t grid_warps() { return (int64_t)STREAM_WARPS_PER_SM * device_sms(); }

}  // namespace

bool stream32_supported(int nu1, int nu2) { return nu1 >= 1 && nu1 <= 3 && nu2 >= 1 && nu2 <= 3; }

cudaError_t launch_stream_down(const BatchLevel<float>* lv, int level, int m, int n, int nu, bool gs, double w,
                               bool zero_c, cudaStream_t s)
{
    const StreamCut cut = down_cut(level, m, n, nu, grid_warps());
    return down(nullptr, cut.nb * cut.strips, cut, lv, nullptr, nu, gs, w, zero_c, s);
}

cudaError_t launch_stream_up(const BatchLevel<float>* lv, int level, int m, int n, int nu, bool gs, double w,
                             cudaStream_t s, double* psi, int64_t psi_pitch)
{
    const StreamCut cut = up_cut(level, m, n, nu, grid_warps());
    return up(nullptr, cut.nb * cut.strips, cut, lv, nullptr, nu, gs, w, psi, psi_pitch, nullptr, s);
}

void stream32_items(int level, int m, int n, int nu1, int nu2, int64_t warps, std::vector<StreamItem>* down_items,
                    std::vector<StreamItem>* up_items)
{
    const StreamCut d = down_cut(level, m, n, nu1, warps), u = up_cut(level, m, n, nu2, warps);
    for (int k = 0; k < d.nb * d.strips; ++k) down_items->push_back(stream_piece(d, k));
    for (int k = 0; k < u.nb * u.strips; ++k) up_items->push_back(stream_piece(u, k));
}

cudaError_t launch_b_stream_down(const StreamItem* items, int count, const BatchLevel<float>* lv,
                                 const int* active, int nu, bool gs, double w, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    return down(items, count, StreamCut{}, lv, active, nu, gs, w, true, s);
}

cudaError_t launch_b_stream_up(const StreamItem* items, int count, const BatchLevel<float>* lv,
                               const int* active, int nu, bool gs, double w, cudaStream_t s,
                               const BatchLevel<double>* lv64)
{
    if (count == 0) return cudaSuccess;
    return up(items, count, StreamCut{}, lv, active, nu, gs, w, nullptr, 0, lv64, s);
}

}  // namespace lap
