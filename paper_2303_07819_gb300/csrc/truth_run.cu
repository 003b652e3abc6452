// truth_run.cu -- up to TRUTH_CHUNK steps of the un-localised DEM (Sec. 4) in
// one cooperative launch, FP32 and FP64.
//
// What bounded it: nine launches a step (clear, bin, three-pass scan, scatter,
// sort, contacts) to find again contacts that last many steps, and in the
// contact kernel the latency of bin -> index -> partner loads.  A floe moves a
// metre a step against radii of hundreds, so it keeps a candidate list, its
// partners within r_l + s_l + r_j + s_j (s: the floe's skin), until some floe
// has moved farther than its skin; a step is then one pass over the lists and
// one grid barrier.  A rebuild costs four barriers: count, block sums, starts,
// scatter (positions and reaches copied in bin order, so a search reads
// consecutive memory), search.
//
// Lists are in ascending floe order and hold every floe that can touch, so a
// floe's force is the sum over its contacts in ascending partner order
// whenever the lists were built: splitting a run of steps differently, or
// resuming it, changes no bit.  Floes of radius <= r_split and larger ones sit
// in separate grids of bins, as the host chose them (setup_truth_bins).
//
// A skin has an upper bound (TruthBins::skin_max), so that lists stay a few
// neighbours long at any speed, and a floe with more candidates than its list
// holds is searched by its warp at every step (next_portion).
//
// Measured, us a step as nine launches and here (FP32): 65,341 power-law floes
// in long runs 65 and 7.9, in calls of one step, with the build, 76 and 77;
// 65,000 floes of 100-300 m with one of 9 or 19 km (125 or 265 partners), in
// calls of 20, 93 and 23 or 189 and 41; 500 floes in a million bins, in calls
// of one step, 61 and 52; 115,200 floes of one size in long runs 9.6.  FP64,
// the power-law floes: 519 and 70, in calls of one step 535 and 138.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cooperative_groups.h>
#include <type_traits>

#include "common.cuh"
#include "truth_step.cuh"

namespace cg = cooperative_groups;

namespace msd {

namespace {

constexpr int TT = 256;       // threads per block
constexpr int LT = 64;        // candidates per floe; the warp searches the bins of a floe with more at every step
constexpr int FOUND = 256;    // touching partners such a search holds

// a floe in the working copy: what a contact test reads, and the rest
struct A32 { uint32_t x, y; float r, h; };
struct A64 { double x, y, r, h; };
template <class R> struct Rest { R u, v, w, th; };

struct Tr32 {
    using R = float;
    using A = A32;
    using State = DevState32;
};
struct Tr64 {
    using R = double;
    using A = A64;
    using State = DevState64;
};

struct Sorted { uint32_t x, y; float reach; int l; };   // a floe in bin order

template <class T>
struct Work {
    typename T::A *A[2];
    Rest<typename T::R> *B[2];
    int *binof, *rank, *cnt, *list;    // [n], [n], [n], [LT][n]
    uint2 *xb;                         // [n] position at the build, fixed point of the domain
    float *skin;                       // [n]
    Sorted *sorted;                    // [n]
    int *bsum;                         // [gridDim]
    int *ctl;                          // flags [3], largest skin [2], sum of speeds [2] (float bits)
    double2 *wind;                     // [TRUTH_CHUNK]
    double2 *tile;                     // FP64: [ty][tx][n_modes] cos, sin of each mode at the tiles' centres
    int tx, ty;                        // 0: no table
};

__device__ __forceinline__ A32 load_a(const DevState32 &s, long long l) { return {s.xq[l], s.yq[l], s.r[l], s.h[l]}; }
__device__ __forceinline__ A64 load_a(const DevState64 &s, long long l) { return {s.x[l], s.y[l], s.r[l], s.h[l]}; }
__device__ __forceinline__ void store_xy(const DevState32 &s, long long l, const A32 &a) { s.xq[l] = a.x; s.yq[l] = a.y; }
__device__ __forceinline__ void store_xy(const DevState64 &s, long long l, const A64 &a) { s.x[l] = a.x; s.y[l] = a.y; }

// 32-bit fixed point of the domain
__device__ __forceinline__ uint2 fixed(const A32 &a, const Geom &) { return make_uint2(a.x, a.y); }
__device__ __forceinline__ uint32_t fixed1(double x, double L)
{
    const double q = floor(x / L * 4294967296.0);
    return (uint32_t)(long long)fmin(fmax(q, 0.0), 4294967295.0);   // a wall's own coordinate is L
}
__device__ __forceinline__ uint2 fixed(const A64 &a, const Geom &g)
{
    return make_uint2(fixed1(a.x, g.Lx), fixed1(a.y, g.Ly));
}

// Is the floe anywhere in the domain?  An FP64 position is not once it is NaN,
// or so far off (above 1e15 domains in a step) that its remainder has no
// digit left: all such floes would lie in the bins at the domain's edge, each
// a candidate of all others.  A fixed-point position always is.
__device__ __forceinline__ bool placed(const A32 &, const Geom &) { return true; }
__device__ __forceinline__ bool placed(const A64 &a, const Geom &g)
{
    return a.x >= 0.0 && a.x <= g.Lx && a.y >= 0.0 && a.y <= g.Ly;
}

// fixed-point separation in metres: the periodic minimum image, or between
// walls the plain difference
__device__ __forceinline__ float sep_x(uint32_t a, uint32_t b, float sx, bool walls)
{
    return walls ? (float)((long long)a - (long long)b) * sx : (float)(int)(a - b) * sx;
}

__device__ __forceinline__ int fbin(uint32_t q, int nb) { return (int)(((unsigned long long)q * (unsigned)nb) >> 32); }

// Calls f(first, last + 1) for the ranges of sorted floes in the bins of one
// grid (nbx x nby bins from bin `base`) within (rx, ry) bin sides of the bin
// that holds a floe at fixed point q, until f returns false (then so does this); bins side by
// side in x are one range.
template <class F>
__device__ __forceinline__ bool visit_ranges(const int *start, int base, int nbx, int nby, uint2 q, float rx, float ry,
                                             bool walls, F &&f)
{
    // margin against rounding
    const int kx = rx * 1.0001f < (float)nbx ? (int)ceilf(rx * 1.0001f) : nbx;
    const int ky = ry * 1.0001f < (float)nby ? (int)ceilf(ry * 1.0001f) : nby;
    const int bx = fbin(q.x, nbx), by = fbin(q.y, nby);
    const bool allx = 2 * kx + 1 >= nbx, ally = 2 * ky + 1 >= nby;
    const int rows = ally ? nby : 2 * ky + 1;
    for (int i = 0; i < rows; i++) {
        int cy = ally ? i : by - ky + i;
        cy = cy < 0 ? cy + nby : (cy >= nby ? cy - nby : cy);
        const int *row = start + base + cy * nbx;
        if (allx) {
            if (!f(row[0], row[nbx])) return false;
            continue;
        }
        const int lo = bx - kx, hi = bx + kx;
        if (!f(row[max(lo, 0)], row[min(hi, nbx - 1) + 1])) return false;
        if (!walls) {
            if (lo < 0 && !f(row[lo + nbx], row[nbx])) return false;
            if (hi >= nbx && !f(row[0], row[hi - nbx + 1])) return false;
        }
    }
    return true;
}

// ascending sort of v[0..N) in registers (bitonic, every index static)
template <int N>
__device__ __forceinline__ void sort_net(int (&v)[N])
{
#pragma unroll
    for (int k = 2; k <= N; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int i = 0; i < N; i++) {
                const int o = i ^ j;
                if (o > i) {
                    const int a = v[i], b = v[o];
                    const bool up = (i & k) == 0;
                    v[i] = up ? min(a, b) : max(a, b);
                    v[o] = up ? max(a, b) : min(a, b);
                }
            }
}

// (not inlined: the registers are the sort's own)
template <int N>
__device__ __noinline__ void sort_list(int *list, long long n, int cnt)
{
    int v[N];
#pragma unroll
    for (int i = 0; i < N; i++) v[i] = i < cnt ? list[i * n] : INT_MAX;
    sort_net(v);
#pragma unroll
    for (int i = 0; i < N; i++)
        if (i < cnt) list[i * n] = v[i];
}

// separation of partner a from floe o in the state's own precision
__device__ __forceinline__ void pair_xy(const A32 &a, const A32 &o, const TruthArgs &t, bool walls, float &dx, float &dy)
{
    dx = sep_x(a.x, o.x, t.k.sx, walls);
    dy = (float)(int)(a.y - o.y) * t.k.sy;
}
__device__ __forceinline__ void pair_xy(const A64 &a, const A64 &o, const TruthArgs &t, bool walls, double &dx, double &dy)
{
    dx = a.x - o.x;
    dy = a.y - o.y;
    if (!walls) dx -= t.g.Lx * rint(dx * t.iLx);
    dy -= t.g.Ly * rint(dy * t.iLy);
}

// the current at a floe: FP32 from the phases in cycles per domain
__device__ __forceinline__ void ocean_at(const Phys<float> &P, const Work<Tr32> &, const TruthArgs &, const A32 &a,
                                         float &uo, float &vo, float &zeta)
{
    const float xf = (float)a.x * INV2_32F, yf = (float)a.y * INV2_32F;
    uo = P.uo_x; vo = P.uo_y; zeta = 0.0f;
    for (int m = 0; m < P.n_modes; m++) {
        float cyc = P.kdx[m] * xf + P.kdy[m] * yf + P.mCyc[m];
        cyc -= floorf(cyc);
        float s, c;
        sincospif(2.0f * cyc, &s, &c);
        uo -= P.mAu[m] * c;
        vo += P.mAv[m] * c;
        zeta -= P.mAz[m] * s;
    }
}

// FP64: each mode's sine and cosine at the centre of the floe's tile turned by
// the angle to the floe, at most a quarter radian, by Taylor sums (remainder
// below 2^-56): 13 FP64 operations where a sincos takes about 60.  Which
// tile, and so the rounding, is a matter of the position alone.
__device__ __forceinline__ void ocean_at(const Phys<double> &P, const Work<Tr64> &w, const TruthArgs &t, const A64 &a,
                                         double &uo, double &vo, double &zeta)
{
    if (w.tx == 0) {
        ocean_f64(P, a.x, a.y, uo, vo, zeta);
        return;
    }
    const int ix = min((int)(a.x * t.iLx * w.tx), w.tx - 1), iy = min((int)(a.y * t.iLy * w.ty), w.ty - 1);
    const double dx = a.x - (ix + 0.5) * (t.g.Lx / w.tx), dy = a.y - (iy + 0.5) * (t.g.Ly / w.ty);
    const double2 *ref = w.tile + ((size_t)max(iy, 0) * w.tx + max(ix, 0)) * P.n_modes;
    uo = P.uo_x; vo = P.uo_y; zeta = 0.0;
    for (int m = 0; m < P.n_modes; m++) {
        const double th = P.mKx[m] * dx + P.mKy[m] * dy, t2 = th * th;
        const double2 r = ref[m];
        double ps = fma(t2, fma(t2, fma(t2, fma(t2, -1.0 / 39916800.0, 1.0 / 362880.0), -1.0 / 5040.0), 1.0 / 120.0),
                        -1.0 / 6.0);
        ps = fma(ps * t2, th, th);
        double pc = fma(t2, fma(t2, fma(t2, fma(t2, fma(t2, 1.0 / 479001600.0, -1.0 / 3628800.0), 1.0 / 40320.0),
                                        -1.0 / 720.0), 1.0 / 24.0), -0.5);
        pc = fma(pc, t2, 1.0);
        const double c = r.x * pc - r.y * ps, s = r.y * pc + r.x * ps;
        uo -= P.mAu[m] * c;
        vo += P.mAv[m] * c;
        zeta -= P.mAz[m] * s;
    }
}

// |(x, y)| of the drag.  In FP64 the rounding is written out: which of the two
// squares the compiler fuses depends on the code around it, and the last bits
// of every floe with it.
__device__ __forceinline__ float length(float x, float y) { return sqrtf(x * x + y * y); }
__device__ __forceinline__ double length(double x, double y) { return sqrt(__fma_rn(x, x, __dmul_rn(y, y))); }

__global__ void k_truth_tiles(Phys<double> P, Geom g, Work<Tr64> w)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= w.tx * w.ty * P.n_modes) return;
    const int m = i % P.n_modes, tile = i / P.n_modes;
    const double x = (tile % w.tx + 0.5) * (g.Lx / w.tx), y = (tile / w.tx + 0.5) * (g.Ly / w.ty);
    double s, c;
    sincos(P.mKx[m] * x + P.mKy[m] * y + P.mPh[m], &s, &c);
    w.tile[i] = make_double2(c, s);
}

// tiles small enough that no mode turns by more than 1/8 from a tile's centre
// along either axis (none if that takes more than 64 MB)
void tile_counts(const Phys<double> &P, const Geom &g, int &tx, int &ty)
{
    double ax = 0.0, ay = 0.0;
    for (int m = 0; m < P.n_modes; m++) {
        ax = fmax(ax, fabs(P.mKx[m]) * g.Lx);
        ay = fmax(ay, fabs(P.mKy[m]) * g.Ly);
    }
    const double nx = ceil(4.0 * ax) + 1.0, ny = ceil(4.0 * ay) + 1.0;
    const bool fits = P.n_modes > 0 && nx * ny * P.n_modes <= 4194304.0;
    tx = fits ? (int)nx : 0;
    ty = fits ? (int)ny : 0;
}

__device__ __forceinline__ void wall_force(const A32 &a, const TruthArgs &t, float u, float v, float w, const Phys<float> &P,
                                           float &fx, float &fy, float &tq, unsigned &deep)
{
    // distances to the walls from the fixed point: exact integers, one rounding
    wall_add((float)a.x * t.k.sx, (float)(4294967296ll - (long long)a.x) * t.k.sx, u, v, w, a.r, a.h, P, fx, fy, tq, deep);
}
__device__ __forceinline__ void wall_force(const A64 &a, const TruthArgs &t, double u, double v, double w,
                                           const Phys<double> &P, double &fx, double &fy, double &tq, unsigned &deep)
{
    wall_add(a.x, t.g.Lx - a.x, u, v, w, a.r, a.h, P, fx, fy, tq, deep);
}

// forward Euler on the position; reading: a centre that would pass a wall
// stays on it (in a stable run the wall's contact force stops the floe long
// before)
__device__ __forceinline__ A32 moved(const A32 &a, const TruthArgs &t, bool walls, float u, float v)
{
    A32 b = a;
    const float dt = t.k.dt;
    if (walls) {
        long long xn = (long long)a.x + __float2int_rn(dt * u * t.k.isx);
        xn = xn < 0 ? 0 : (xn > 4294967295ll ? 4294967295ll : xn);
        b.x = (uint32_t)xn;
    } else {
        b.x = a.x + (uint32_t)__float2int_rn(dt * u * t.k.isx);
    }
    b.y = a.y + (uint32_t)__float2int_rn(dt * v * t.k.isy);
    return b;
}
__device__ __forceinline__ A64 moved(const A64 &a, const TruthArgs &t, bool walls, double u, double v)
{
    A64 b = a;
    b.x = a.x + t.dt * u;
    b.y = a.y + t.dt * v;
    if (walls) b.x = fmin(fmax(b.x, 0.0), t.g.Lx);
    else if (!(b.x >= 0.0 && b.x < t.g.Lx)) b.x -= t.g.Lx * floor(b.x / t.g.Lx);
    if (!(b.y >= 0.0 && b.y < t.g.Ly)) b.y -= t.g.Ly * floor(b.y / t.g.Ly);
    return b;
}

// A floe's reach: its radius, its skin and what covers the rounding of the
// FP32 tests (negative: a floe that is nowhere touches none).
template <class A>
__device__ __forceinline__ float reach_of(const A &p, float skin, const Geom &g)
{
    return placed(p, g) ? ((float)p.r + skin) * 1.00001f + 1.0e-9f * fmaxf((float)g.Lx, (float)g.Ly) : -FLT_MAX;
}

// Calls f(first, last + 1) for the ranges of w.sorted that hold every floe
// within reach of one at build position x with reach `own`, until f returns
// false; smax: the largest skin.
template <class T, class F>
__device__ __forceinline__ void near_ranges(const Work<T> &w, const TruthArgs &a, const TruthBins &tb, uint2 x, float own,
                                            float smax, F &&f)
{
    const bool walls = a.g.walls != 0;
    const float Lx = (float)a.g.Lx, Ly = (float)a.g.Ly;
    const float r1 = own + (tb.r_split + smax) * 1.00001f, r2 = own + (tb.r_max + smax) * 1.00001f;
    if (visit_ranges(tb.start, 0, tb.nbx, tb.nby, x, r1 * tb.nbx / Lx, r1 * tb.nby / Ly, walls, f) && tb.nbx2 > 0)
        visit_ranges(tb.start, tb.nbx * tb.nby, tb.nbx2, tb.nby2, x, r2 * tb.nbx2 / Lx, r2 * tb.nby2 / Ly, walls, f);
}

// were the two floes within reach at the build?
template <class T>
__device__ __forceinline__ bool in_reach(const Sorted &q, uint2 x, float own, const TruthArgs &a)
{
    constexpr bool unplaced = std::is_same<T, Tr64>::value;      // may a reach be negative?
    const float dx = sep_x(q.x, x.x, a.k.sx, a.g.walls != 0), dy = (float)(int)(q.y - x.y) * a.k.sy, r = own + q.reach;
    return !(dx * dx + dy * dy >= r * (unplaced ? fabsf(r) : r));
}

// the warp's numbers v[0..m), all different, into ascending order (m <= FOUND)
__device__ __forceinline__ void sort_warp(int *v, int m)
{
    const int lane = threadIdx.x & 31;
    int x[FOUND / 32], rank[FOUND / 32];
    __syncwarp();
#pragma unroll
    for (int k = 0; k < FOUND / 32; k++) {
        x[k] = lane + 32 * k < m ? v[lane + 32 * k] : 0;
        rank[k] = 0;
    }
    for (int i = 0; i < m; i++) {
        const int o = v[i];
#pragma unroll
        for (int k = 0; k < FOUND / 32; k++) rank[k] += o < x[k] ? 1 : 0;
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < FOUND / 32; k++)
        if (lane + 32 * k < m) v[rank[k]] = x[k];
    __syncwarp();
}

// Floes with more candidates than a list holds, of one warp's 32: their
// contacts are found by the whole warp, a candidate a lane, and handed to the
// floe's lane in portions of up to LT, in ascending order.  (One lane
// searching for one contact after another: 157 us a step for the floe of 19 km
// above, 41 so.)
struct LongLists {
    unsigned left;         // lanes whose floes are still to be searched
    int src, at, held;     // the floe's lane; the next partner to hand on, partners found
    int above;             // its partners up to this one are done with
    int more;              // are there more than were held?
    int found[FOUND];
};

// The next portion into the list of its floe: to the floe's lane the number of
// partners, 0 to the others, -1 to all if there is none left.  l0: the floe
// of lane 0.  (Not inlined: its registers are its own.)
template <class T>
__device__ __noinline__ int next_portion(const Work<T> &w, const TruthArgs &a, const TruthBins &tb,
                                         const typename T::A *A, long long l0, float smax, LongLists &S)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    __syncwarp();
    unsigned left = S.left;
    int src = S.src, at = S.at, held = S.held, above = S.above, more = S.more;
    __syncwarp();
    while (at == held) {
        if (!more) {
            if (left == 0u) return -1;
            src = __ffs((int)left) - 1;
            left &= left - 1u;
            above = -1;
        }
        const int l = (int)l0 + src;
        const typename T::A me = A[l];
        const uint2 x = w.xb[l];
        const float own = reach_of(me, w.skin[l], a.g);
        const bool walls = a.g.walls != 0;
        int m = 0, lim = INT_MAX;
        near_ranges<T>(w, a, tb, x, own, smax, [&](int i0, int i1) {
            for (; i0 < i1; i0 += 32) {
                bool hit = false;
                int j = 0;
                if (i0 + lane < i1) {
                    const Sorted q = w.sorted[i0 + lane];
                    j = q.l;
                    if (j != l && j > above && j < lim && in_reach<T>(q, x, own, a)) {
                        typename T::R dx, dy;
                        const typename T::A o = A[j];
                        pair_xy(o, me, a, walls, dx, dy);
                        const typename T::R r = me.r + o.r;
                        hit = dx * dx + dy * dy < r * r * typename T::R(1.00001);   // the walk decides
                    }
                }
                const unsigned hits = __ballot_sync(FULL, hit);
                if (hit) S.found[m + __popc(hits & ((1u << lane) - 1u))] = j;
                m += __popc(hits);
                if (m > FOUND - 32) {      // the smaller half, and from here on only what belongs among it
                    sort_warp(S.found, m);
                    m = FOUND / 2;
                    lim = S.found[m];
                    __syncwarp();          // (read by all before the next is put there)
                }
            }
            return true;
        });
        sort_warp(S.found, m);
        more = lim != INT_MAX;
        at = 0;
        held = m;
        if (more) above = lim - 1;
    }
    const int k = min(LT, held - at);
    for (int i = lane; i < k; i += 32) w.list[i * a.n + l0 + src] = S.found[at + i];
    if (lane == 0) {
        S.left = left;
        S.src = src;
        S.at = at + k;
        S.held = held;
        S.above = above;
        S.more = more;
    }
    __syncwarp();
    return lane == src ? k : 0;
}

// exclusive scan of one value per thread over the block; total to all threads
__device__ __forceinline__ int block_excl(int v, int *ws, int &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    __syncthreads();
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    int base = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < TT / 32; w++) {
        base += w < warp ? ws[w] : 0;
        total += ws[w];
    }
    return base + x - v;
}

template <class T>
__global__ void __launch_bounds__(TT)
k_truth_run(typename T::State in, typename T::State out, Phys<typename T::R> P, const __grid_constant__ TruthArgs a,
            const __grid_constant__ TruthBins tb, const __grid_constant__ Work<T> w, int nsteps)
{
    using R = typename T::R;
    using A = typename T::A;
    cg::grid_group grid = cg::this_grid();
    __shared__ int ws[TT / 32];
    __shared__ float wmax[TT / 32], wsum[TT / 32];
    __shared__ LongLists longs[TT / 32];
    const long long n = a.n, gt = blockIdx.x * (long long)TT + threadIdx.x, gs = gridDim.x * (long long)TT;
    const bool walls = a.g.walls != 0;
    const int nbins = tb.nbins(), nb1 = tb.nbx * tb.nby;
    const float sx = a.k.sx, sy = a.k.sy;
    R *fd = reinterpret_cast<R *>(a.fd);
    unsigned long long ndeep = 0;
    bool bad = false;

    // a floe's speed as the skins count it: at most what fills the widest skin
    // (NaN too)
    auto speed_of = [&](float u, float v) { return fminf(sqrtf(u * u + v * v), tb.skin_max / (48.0f * (float)a.dt)); };
    // a sum of the floes' speeds over the grid into ctl[at]; the order of its
    // additions varies, and with it the skins, but no result
    auto add_speeds = [&](float vs, int at) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) vs += __shfl_xor_sync(0xffffffffu, vs, d);
        if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = vs;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int i = 1; i < TT / 32; i++) vs += wsum[i];
            atomicAdd(reinterpret_cast<float *>(&w.ctl[at]), vs);
        }
    };
    float vs0 = 0.0f;
    for (long long l = gt; l < n; l += gs) {
        w.A[0][l] = load_a(in, l);
        w.B[0][l] = {in.u[l], in.v[l], in.w[l], in.th[l]};
        vs0 += speed_of((float)in.u[l], (float)in.v[l]);
    }
    for (long long i = gt; i < nbins; i += gs) tb.count[i] = 0;
    for (long long i = gt; i < nsteps; i += gs) {
        R ua, va;
        wind_at(P, (double)(a.step + i) * a.dt, ua, va);
        w.wind[i] = make_double2((double)ua, (double)va);
    }
    if (gt < 3) w.ctl[gt] = gt == 2 ? 1 : 0;      // step -1 asks step 0 for lists
    if (gt >= 3 && gt < 7) w.ctl[gt] = 0;
    grid.sync();
    add_speeds(vs0, 5 + 1);       // for the first build
    grid.sync();

    int cur = 0, par = 0;
    for (int s = 0; s < nsteps; s++) {
        const bool need = *(volatile int *)&w.ctl[(s + 2) % 3] != 0;
        if (gt == 0) w.ctl[(s + 1) % 3] = 0;      // read at the last step, written at the next
        if (need) {
            // count the floes of each bin; skins: 48 steps' way (in a launch's last
            // twelve, four times what is left: a call of one step needs no longer
            // lists) at the current speed, or at half the mean one (at the build
            // before), plus 2 % of the radius, none wider than skin_max: a fast floe
            // leaves its skin sooner, and a state that diverges keeps lists of
            // bounded length
            float smax = 0.0f, vsum = 0.0f;
            const float ahead = (float)a.dt * (float)min(48, 4 * (nsteps - s));
            const float vfloor = 0.5f * __int_as_float(*(volatile int *)&w.ctl[5 + (par ^ 1)]) / (float)n;
            for (long long l = gt; l < n; l += gs) {
                const A p = w.A[cur][l];
                const Rest<R> q = w.B[cur][l];
                const uint2 x = fixed(p, a.g);
                const float r = (float)p.r, speed = speed_of((float)q.u, (float)q.v);
                vsum += speed;
                const float skin = fminf(ahead * fmaxf(speed, vfloor), tb.skin_max) + 0.02f * r;
                w.skin[l] = skin;
                w.xb[l] = x;
                smax = fmaxf(smax, skin);
                const int b = r <= tb.r_split ? fbin(x.y, tb.nby) * tb.nbx + fbin(x.x, tb.nbx)
                                              : nb1 + fbin(x.y, tb.nby2) * tb.nbx2 + fbin(x.x, tb.nbx2);
                w.binof[l] = b;
                w.rank[l] = atomicAdd(&tb.count[b], 1);
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, d));
            if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = smax;
            __syncthreads();
            if (threadIdx.x == 0) {
                for (int i = 1; i < TT / 32; i++) smax = fmaxf(smax, wmax[i]);
                atomicMax(&w.ctl[3 + par], __float_as_int(smax));   // skins are positive: ordered as integers
            }
            add_speeds(vsum, 5 + par);
            grid.sync();
            // each warp a run of bins, a bin a lane: the blocks' totals, then the
            // starts
            const int per = ((nbins + (int)gridDim.x * (TT / 32) - 1) / ((int)gridDim.x * (TT / 32)) + 31) & ~31;
            const int c0 = (int)min((long long)(blockIdx.x * (TT / 32) + (threadIdx.x >> 5)) * per, (long long)nbins);
            const int c1 = min(c0 + per, nbins), lane = threadIdx.x & 31;
            int sum = 0;
            for (int i = c0 + lane; i < c1; i += 32) sum += tb.count[i];
            int total;
            const int mine = block_excl(sum, ws, total);
            if (threadIdx.x == 0) w.bsum[blockIdx.x] = total;
            if (gt == 0) w.ctl[3 + (par ^ 1)] = w.ctl[5 + (par ^ 1)] = 0;   // the next build's sums
            grid.sync();
            int before = 0;
            for (int i = threadIdx.x; i < (int)blockIdx.x; i += TT) before += w.bsum[i];
            block_excl(before, ws, before);
            int run = before + __shfl_sync(0xffffffffu, mine, 0);
            for (int i0 = c0; i0 < c1; i0 += 32) {
                const int c = i0 + lane < c1 ? tb.count[i0 + lane] : 0;
                int x = c;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, x, d);
                    if (lane >= d) x += y;
                }
                if (i0 + lane < c1) {
                    tb.start[i0 + lane] = run + x - c;
                    tb.count[i0 + lane] = 0;
                }
                run += __shfl_sync(0xffffffffu, x, 31);
            }
            grid.sync();
            for (long long l = gt; l < n; l += gs) {
                const uint2 x = w.xb[l];
                const float reach = reach_of(w.A[cur][l], w.skin[l], a.g);
                w.sorted[tb.start[w.binof[l]] + w.rank[l]] = {x.x, x.y, reach, (int)l};
            }
            grid.sync();
        }
        // the largest skin of the lists in use (of either parity's build)
        if (need) par ^= 1;
        const float smax = __int_as_float(*(volatile int *)&w.ctl[3 + (par ^ 1)]);
        if (need) {
            for (long long l = gt; l < n; l += gs) {
                int c = 0;
                const A p = w.A[cur][l];
                const uint2 x = w.xb[l];
                const float own = reach_of(p, w.skin[l], a.g);
                if (placed(p, a.g))
                    near_ranges<T>(w, a, tb, x, own, smax, [&](int i0, int i1) {
                        for (int i = i0; i < i1 && c <= LT; i++) {   // (one more than a list holds is all there is to know)
                            const Sorted q = w.sorted[i];
                            if (q.l == (int)l || !in_reach<T>(q, x, own, a)) continue;
                            if (c < LT) w.list[c * n + l] = q.l;
                            c++;
                        }
                        return c <= LT;
                    });
                w.cnt[l] = c;
                if (c > 1 && c <= 16) sort_list<16>(w.list + l, n, c);
                else if (c > 16 && c <= LT) sort_list<LT>(w.list + l, n, c);
            }
        }
        const bool last = s == nsteps - 1;
        const double2 wa = w.wind[s];
        bool far = false;
        for (long long l0 = gt - (threadIdx.x & 31); l0 < n; l0 += gs) {      // a warp's 32 floes
            const bool valid = l0 + (threadIdx.x & 31) < n;
            const long long l = valid ? l0 + (threadIdx.x & 31) : l0;
            const A me = w.A[cur][l];
            const Rest<R> q = w.B[cur][l];
            R fx = 0, fy = 0, tq = 0;
            unsigned deep = 0;
            int c = valid ? w.cnt[l] : 0;
            const bool any_long = __any_sync(0xffffffffu, c > LT);
            if (any_long) {
                const unsigned left = __ballot_sync(0xffffffffu, c > LT);
                if ((threadIdx.x & 31) == 0) {
                    LongLists &S = longs[threadIdx.x >> 5];
                    S.left = left;
                    S.at = S.held = S.more = 0;
                }
                if (c > LT) c = 0;
            }
            // the floe's list, contacts in ascending partner order (the portions of a
            // long one take the same way, so its forces are rounded alike)
            do {
                for (int i = 0; i < c; i += 4) {      // four partners' loads in flight
                    int j[4];
                    A o[4];
#pragma unroll
                    for (int k = 0; k < 4; k++) j[k] = w.list[min(i + k, c - 1) * n + l];
#pragma unroll
                    for (int k = 0; k < 4; k++) o[k] = w.A[cur][j[k]];
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        if (i + k >= c) continue;
                        R dx, dy;
                        pair_xy(o[k], me, a, walls, dx, dy);
                        const R d2 = dx * dx + dy * dy, S = me.r + o[k].r;
                        if (d2 < S * S) {
                            const Rest<R> p = w.B[cur][j[k]];
                            contact_add(dx, dy, d2, me.r, o[k].r, me.h, o[k].h, p.u - q.u, p.v - q.v, q.w, p.w, P, fx, fy,
                                        tq, deep);
                        }
                    }
                }
                if (any_long) c = next_portion<T>(w, a, tb, w.A[cur], l0, smax, longs[threadIdx.x >> 5]);
            } while (any_long && c >= 0);
            if (!valid) continue;
            R uo, vo, zeta;
            ocean_at(P, w, a, me, uo, vo, zeta);
            if (walls) wall_force(me, a, q.u, q.v, q.w, P, fx, fy, tq, deep);
            R Fdx, Fdy, Td;
            drag_force(P, uo, vo, zeta, (R)wa.x, (R)wa.y, q.u, q.v, q.w, me.r, Fdx, Fdy, Td,
                       [](R x, R y) { return length(x, y); });
            fx += Fdx; fy += Fdy; tq += Td;
            const R dt = (R)a.dt;
            const R m = P.mass_c * me.r * me.r * me.h;
            const R I = P.inertia_f * m * me.r * me.r;
            const A to = moved(me, a, walls, q.u, q.v);
            const Rest<R> v = {q.u + dt * (fx / m), q.v + dt * (fy / m), q.w + dt * (tq / I), q.th + dt * q.w};
            bad |= !(isfinite(v.u) && isfinite(v.v) && isfinite(v.w));
            ndeep += deep ? 1u : 0u;
            if (last) {
                store_xy(out, l, to);
                out.u[l] = v.u;
                out.v[l] = v.v;
                out.w[l] = v.w;
                out.th[l] = v.th;
                out.r[l] = me.r;
                out.h[l] = me.h;
                fd[l] = Fdx; fd[n + l] = Fdy; fd[2 * n + l] = Td;
            } else {
                w.A[cur ^ 1][l] = to;
                w.B[cur ^ 1][l] = v;
                const uint2 x = fixed(to, a.g), x0 = w.xb[l];
                const float bx = sep_x(x.x, x0.x, sx, walls), by = (float)(int)(x.y - x0.y) * sy, sk = w.skin[l];
                far |= !(bx * bx + by * by <= sk * sk);
            }
        }
        if (last) break;
        if (__syncthreads_or(far) && threadIdx.x == 0) w.ctl[s % 3] = 1;
        grid.sync();
        cur ^= 1;
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(&a.ctrl->err, ERR_NONFINITE);
    if (ndeep) atomicAdd(&a.ctrl->deep, ndeep);
}

// Blocks for n floes or, in sparse ice, for a bin of every 32 to a thread: a
// build goes over all bins (500 floes of 50 m in 100 km, a million bins, a call
// of one step: 2650 us on the two blocks of their floes, 52 so; blocks for a
// bin of every 8 to a thread: 52, but 4.5 us a step in long runs instead of 4.1).
template <class T>
int grid_of(long long n, int nbins)
{
    // (made by the first caller; others wait for it)
    static const long long most = [] {
        int dev = 0, nsm = 0, b = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_truth_run<T>, TT, 0) != cudaSuccess) b = 0;
        return (long long)std::max(b, 1) * nsm;
    }();
    const long long need = (std::max<long long>(n, nbins / 32) + TT - 1) / TT;
    return (int)(need < 1 ? 1 : (need < most ? need : most));
}

// the work arrays in one allocation of `bytes` (base NULL: only its size)
template <class T>
Work<T> carve(unsigned char *base, long long n, const Phys<double> &P, const Geom &g, size_t &bytes)
{
    size_t o = 0;
    auto take = [&](auto *&p, size_t count) {
        using E = std::remove_reference_t<decltype(*p)>;
        p = reinterpret_cast<E *>(base + o);
        o += (sizeof(E) * count + 255) & ~size_t(255);
    };
    Work<T> w{};
    const bool wide = sizeof(typename T::R) == 8;
    for (int k = 0; k < 2; k++) {
        take(w.A[k], n);
        take(w.B[k], n);
    }
    take(w.binof, n);
    take(w.rank, n);
    take(w.cnt, n);
    take(w.list, (size_t)LT * n);
    take(w.xb, n);
    take(w.skin, n);
    take(w.sorted, n);
    take(w.bsum, 4096);
    take(w.ctl, 8);
    take(w.wind, TRUTH_CHUNK);
    if (wide) tile_counts(P, g, w.tx, w.ty);
    take(w.tile, (size_t)w.tx * w.ty * P.n_modes);
    bytes = o;
    return w;
}

template <class T>
cudaError_t launch(const typename T::State &in, const typename T::State &out, const Phys<typename T::R> &P,
                   const Phys<double> &P64, const TruthArgs &a, TruthBins &b, void *work, int nsteps, cudaStream_t st)
{
    if (a.n <= 0 || nsteps <= 0) return cudaSuccess;
    size_t bytes;
    Work<T> w = carve<T>(static_cast<unsigned char *>(work), a.n, P64, a.g, bytes);
    typename T::State si = in, so = out;
    Phys<typename T::R> p = P;
    TruthArgs ta = a;
    void *args[] = {&si, &so, &p, &ta, &b, &w, &nsteps};
    return cudaLaunchCooperativeKernel((const void *)k_truth_run<T>, dim3(grid_of<T>(a.n, b.nbins())), dim3(TT), args, 0,
                                       st);
}

}  // namespace

size_t truth_work_bytes(int precision, long long n, const Phys<double> &P, const Geom &g)
{
    size_t bytes = 0;
    if (precision == 1) carve<Tr64>(nullptr, n, P, g, bytes);
    else carve<Tr32>(nullptr, n, P, g, bytes);
    return bytes;
}

cudaError_t truth_work_init(int precision, long long n, const Phys<double> &P, const Geom &g, void *work, cudaStream_t st)
{
    if (precision != 1) return cudaSuccess;
    size_t bytes;
    const Work<Tr64> w = carve<Tr64>(static_cast<unsigned char *>(work), n, P, g, bytes);
    const int k = w.tx * w.ty * P.n_modes;
    if (k > 0) k_truth_tiles<<<(k + 255) / 256, 256, 0, st>>>(P, g, w);
    return cudaGetLastError();
}

cudaError_t launch_truth_run32(const DevState32 &in, const DevState32 &out, const Phys<float> &P, const Phys<double> &P64,
                               const TruthArgs &a, TruthBins &b, void *work, int nsteps, cudaStream_t st)
{
    return launch<Tr32>(in, out, P, P64, a, b, work, nsteps, st);
}

cudaError_t launch_truth_run64(const DevState64 &in, const DevState64 &out, const Phys<double> &P, const TruthArgs &a,
                               TruthBins &b, void *work, int nsteps, cudaStream_t st)
{
    return launch<Tr64>(in, out, P, P, a, b, work, nsteps, st);
}

}  // namespace msd
