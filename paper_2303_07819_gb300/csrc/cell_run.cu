// cell_run.cu -- FP32 msDEM cell steps for a whole run of fine steps in one
// launch, every floe resident in a thread's registers (launch variant 5).
//
// Between two coarse steps a cell depends on nothing but itself (Sec. 3.1:
// each coarse cell carries its own doubly periodic DEM; the gradual-update
// increments of Algorithm 1 are fixed at the coarse step), so a block can
// take its cells through every fine step of a run and touch global memory
// only at the run's two ends.
//
// Work: the cells are packed into groups of at most 256, 512 or 1024 floes: a
// cell of more than 256 or 512 floes is a group of its own, smaller cells share
// groups of the first kind, first fit by decreasing size.  A cell's floes so
// always run the code of its own size class, whatever else the model holds.
// A class is one persistent launch of blocks of as many threads, a floe each,
// that take groups from a ticket queue in decreasing order of work.  A floe's
// state and forcing stay in registers for the run, what a step reads once stays
// in shared memory (64 registers a thread, 1024 threads an SM); per step it
// publishes its position and velocity to shared memory (two buffers, so one
// barrier per step separates the step that reads a buffer from the one that
// writes it again).
//
// What bounds it: the issue of instructions (2.0M floes: the class of 256 by
// itself issues in 72 % of the cycles, the classes side by side reach 87 % of
// the peak rate; no memory traffic to speak of), in steps with few floes a
// group the latency of the chain list -> partner -> force -> barrier, in runs
// of one step the build and the reduction.  Per interval of
// 100 steps, before the candidate lists took their present form (slots of 16
// a floe, a floe with more tested its whole cell; 256 threads with up to four
// floes each; two barriers a step) and now: 65,505 power-law floes 338 -> 279
// us fresh and 1210 -> 380 packed, 115,200 floes of one size 309 -> 264 and
// 529 -> 455, 500,658 floes 1535 -> 890 and 7660 -> 1170, 2.0M floes 2914 ->
// 2580 and 3110 -> 2710, 256 floes 274 -> 190.
//
// Contacts (Eq. 2.2): a floe tests only its candidates, the floes of its
// cell within reach at the last build: r_l G + s_l + r_j G + s_j, with G the
// growth the cell's gradual updates can still give its radii in this
// coarse interval and s_f the floe's own skin (its speed times a horizon of
// steps).  A build is a counting sort of the group's floes into per-cell
// bins (floes whose reach fits half a bin) and a per-cell list of the other,
// "large" floes; every pair is searched from one side and its hit recorded on
// both.  A group builds at the first step of a run and again once a floe has
// moved more than its skin.  The lists of a group lie one after another in one
// pool of LMAX candidates a floe on average, so a large floe with hundreds of
// partners costs what its partners cost; a list of up to LSER is walked by its
// floe's lane, a longer one by the whole warp, a candidate a lane (on packed
// power-law floes the warp otherwise waits for its one large floe: 1210 us an
// interval for the 380 above).  Lists that do not fit are built again with shorter
// skins, and if that does not help every pair of the cell is tested.  Each
// list is sorted by floe index, so a floe always sums its contacts in ascending
// partner order -- the order of the all-pairs loop over (l < j) in cell order,
// whatever the skins, bins or build steps were.
//
// Ocean (Eq. 2.1c-d at the floe's global position): each floe keeps the
// first-order Taylor expansion of the current and its curl about a centre
// near it and evaluates that every step (6 multiply-adds instead of a sum
// of modes).  The neglected term stays below the FP32 rounding of the mode
// sum while the floe is within sqrt(P.ocean_d2) of the centre (the bound is
// derived from the modes' wave numbers on the host); when a floe of a cell
// goes farther, or wraps across its cell's edge, every floe of that cell
// expands again at its current position with the modes' full sums at the
// next step (a decision of the cell alone, whichever cells share its block).
//
// Moments (Algorithm 1): the window needs per step the cell's mass-weighted
// mean velocity and its drag totals.  A gradual update scales the radii of
// all floes of a cell by one factor (Eq. 3.5 with reading c11) and leaves
// thicknesses alone, so each floe's share m_f / M of its cell's mass is the
// same at every step of a coarse interval; then sum_s (sum_f m_f u_f,s) / M
// = sum_f (m_f / M) (sum_s u_f,s).  Each floe sums its velocity and drag
// over the interval and the block reduces these sums once, at the
// interval's end.  A run that ends inside an interval stores the floes'
// running sums and expansion centres (the carry) and the next run picks
// them up, so a coarse interval gives the same result bit for bit however
// it is split into runs (an uncoupled run short of the interval has no carry:
// its floes take new centres every step).  The cell moments of the run's last
// step (all 12 columns) are reduced once at the end.  Reductions are exact
// (integer sums of fixed-point values), so their order does not matter.
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

#include "common.cuh"
#include "fixsum.cuh"

namespace msd {

namespace {

// Tunables (measured on the 128 x 128 batched workload; see the build flags)
#ifndef MS_RUN_LMAX
#define MS_RUN_LMAX 12
#endif
#ifndef MS_RUN_LSER
#define MS_RUN_LSER 24
#endif
#ifndef MS_RUN_K1_BLOCKS
#define MS_RUN_K1_BLOCKS 4
#endif

constexpr int LMAX = MS_RUN_LMAX;  // candidates per floe: slots of a build's first sort, and the mean its pool holds
constexpr int LSER = MS_RUN_LSER;  // longest list a lane walks alone
constexpr int GCMAX = RUN_GCMAX;   // cells per group
constexpr int WIND = 128;          // steps per wind table
constexpr int NRED = 16;           // values per reduction (moment columns 1-11, window sums)
constexpr int NEVT = 16;           // gradual updates per interval with a precomputed radius ratio

template <int RT, int K>
struct RunSm {
    static constexpr int F = RT * K;
    static constexpr int NW = RT / 32;
    static constexpr int PAIRS = LMAX * F;      // candidate pairs of the group's lists
    static constexpr int OV = F > 512 ? 768 : 384;   // hits beyond the floes' LMAX slots a build holds
    struct Buf {                    // what a floe publishes for a step
        float4 A[F];                // u, v, w, h
        uint2 Q[F];                 // fixed-point position
        float R[F];                 // radius
    } buf[2];
    float4 D[F];                    // by thread slot: dt / mass, dt / inertia, squared skin, thickness
    float4 W[F];                    // running window sums of a coupled run: u, v, drag x, y ...
    float WT[F];                    // ... and drag torque
    uint2 B[F];                     // position at the build
    union {
        unsigned short L[LMAX][F];  // build: each floe's first hits, slot-major
        unsigned short V[PAIRS];    // the lists, one after another by thread, ascending
        struct {                    // the run's end
            unsigned long long csum[NRED][GCMAX];   // per-cell sums, fixed point (two's complement)
            int cexp[NRED][GCMAX];  // their binary exponents: the largest of the cell's values
        };
    };
    unsigned OVP[OV];               // build: hits beyond LMAX (floe << 16 | partner)
    union {
        float RE[F];                // build: reach of each floe, r G + s
        int ST[F];                  // build: where the next hit beyond LMAX goes (owner's lane << 16 | place)
    };
    int LC[F];                      // build: list lengths (other floes append)
    unsigned short SF[F];           // floes in bin order (build)
    unsigned short BF[F];           // bin of each floe (build)
    int BS[F + GCMAX + 1];          // bin counts, then starts
    int BC[F + GCMAX + 1];          // bin cursors
    float2 Cm[GCMAX][MAXM];         // per cell and mode: corner phase (cos, sin), or (cycles, -)
    float mode[MAXM][7];            // per mode: turn across a cell in x, y (rad, or cycles); kx, ky; Au, Av, Az
    float rg[2][GCMAX][4];          // gradual update per cell (g, du, dv, dw), by step parity
    float cgrow[GCMAX][NEVT + 1];   // growth the cell's radii can still take this interval, by updates done
    float cdv[GCMAX][NEVT + 1];     // speed the cell's gradual updates can still add, by updates done
    double cwin[GCMAX][NWIN];       // the cells' window sums (loaded at the run's start, stored at its end)
    float rgev[GCMAX][NEVT];        // radius ratio of each gradual update of the interval, per cell
    float2 wind[WIND];
    int cc[GCMAX], cfs[GCMAX], cn[GCMAX], cnb[GCMAX], cbb[GCMAX], cgo[GCMAX];
    int cskip[GCMAX];               // a closure cell: no DEM this interval (its floes stay where they are)
    int4 grp;                       // the group's floes and cells, gradual update on (0 / 1)
    int ncg, nfl, nbin, item, allskip, nov, nbuild, deep;
    int wtot[K][NW];                // build: pairs per warp and row
    float vsum[2];                  // group speed sums of the builds, by build parity
    float hz;                       // horizon of the skins (s; negative: not to be shortened)
    int cflag[3][GCMAX];            // a floe of the cell strayed from its ocean centre, by step mod 3
};

// Segmented warp reductions towards the head of each segment: lanes [lane,
// end) of this warp belong to the caller's segment; after the call the
// segment's first lane holds its maximum or total.  Integer operations, so
// the result does not depend on the order.  A warp whose lanes are one
// segment (`whole`) takes the hardware's reductions, a sum of 32 values of at
// most 2^50 as three 17-bit digits (the last one signed); else `longest` is the
// warp's longest segment, which ends the rounds of shuffles.
__device__ __forceinline__ int seg_max(int x, int lane, int end_lane, bool whole, int longest)
{
    if (whole) return __reduce_max_sync(0xffffffffu, x);
#pragma unroll 1
    for (int d = 1; d < longest; d <<= 1) {
        const int y = __shfl_down_sync(0xffffffffu, x, d);
        if (lane + d < end_lane) x = max(x, y);
    }
    return x;
}

__device__ __forceinline__ long long seg_sum(long long x, int lane, int end_lane, bool whole, int longest)
{
    if (whole) {
        const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)x & 0x1ffffu);
        const unsigned mi = __reduce_add_sync(0xffffffffu, (unsigned)(x >> 17) & 0x1ffffu);
        const int hi = __reduce_add_sync(0xffffffffu, (int)(x >> 34));
        return ((long long)hi << 34) + ((long long)mi << 17) + (long long)lo;
    }
#pragma unroll 1
    for (int d = 1; d < longest; d <<= 1) {
        const long long y = __shfl_down_sync(0xffffffffu, x, d);
        if (lane + d < end_lane) x += y;
    }
    return x;
}

// Exclusive scan of BS[0..nb) in place (block-wide); BC gets a copy of the
// starts.  Ends with a barrier.
template <int RT, int K>
__device__ void block_scan_bins(RunSm<RT, K> &S, int nb)
{
    constexpr int NW = RT / 32;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int per = (nb + RT - 1) / RT;
    const int b0 = t * per, b1 = min(b0 + per, nb);
    int s = 0;
    for (int b = b0; b < b1; b++) s += S.BS[b];
    int x = s;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) S.wtot[0][warp] = x;
    __syncthreads();
    int wbase = 0;
    for (int k = 0; k < NW; k++) wbase += k < warp ? S.wtot[0][k] : 0;
    int run = wbase + x - s;
    for (int b = b0; b < b1; b++) {
        const int c = S.BS[b];
        S.BS[b] = run;
        S.BC[b] = run;
        run += c;
    }
    __syncthreads();
}

// |(a, b)| from the hardware reciprocal square root (within a few ulp of
// the correctly rounded norm; 0 for the zero vector)
__device__ __forceinline__ float fast_norm(float a, float b)
{
    const float q = fmaf(a, a, b * b);
    return q * inv_sqrt(q);
}

// Separation of partner q from the floe at (xq, yq): the cell's periodic
// minimum image by fixed-point wrap-around.
struct PairSep {
    float dx, dy, d2;
};
__device__ __forceinline__ PairSep pair_sep(uint2 q, uint32_t xq, uint32_t yq, float sx, float sy)
{
    PairSep s;
    s.dx = __fmul_rn((float)(int)(q.x - xq), sx);
    s.dy = __fmul_rn((float)(int)(q.y - yq), sy);
    s.d2 = __fmaf_rn(s.dx, s.dx, __fmul_rn(s.dy, s.dy));
    return s;
}
__device__ __forceinline__ bool pair_touch(const PairSep &s, float rl, float rq)
{
    const float sum = __fadd_rn(rl, rq);
    return s.d2 > 0.0f && s.d2 < __fmul_rn(sum, sum);
}

// Has a coordinate wrapped across its cell's edge on the way from x0 to x,
// d = (int)(x - x0)?  Sign bit of the result: the unsigned difference borrows
// (x < x0) where the signed one is not negative, or the other way round.
__device__ __forceinline__ uint32_t wrapped_bit(uint32_t x, uint32_t x0, uint32_t d)
{
    return ((~x & x0) | (~(x ^ x0) & d)) ^ d;
}

// Has a floe at fixed point (xq, yq) left the region where an expansion of
// the current about (x0, y0) holds (squared distance above d2), or wrapped
// across its cell's edge since (its global position jumped by a cell side
// while the fixed-point difference stayed small)?
__device__ __forceinline__ bool ocean_stale(uint32_t xq, uint32_t yq, uint32_t x0, uint32_t y0, float sx, float sy,
                                            float d2)
{
    const uint32_t ix = xq - x0, iy = yq - y0;
    const float dx = (float)(int)ix * sx, dy = (float)(int)iy * sy;
    return (int)(wrapped_bit(xq, x0, ix) | wrapped_bit(yq, y0, iy)) < 0 || dx * dx + dy * dy > d2;
}

// Ocean current and curl, and their gradients (per metre of global X, Y).
struct OceanExp {
    float u, v, z, ux, uy, vx, vy, zx, zy;
};

// The expansion at the fraction (xf, yf) of cell ci: the modes' full sums in
// the FP32 phase-split form (corner phase Cm, turn across the cell).
template <int RT, int K>
__device__ __forceinline__ OceanExp ocean_expand(const Phys<float> &P, const RunSm<RT, K> &S, int ci, float xf, float yf,
                                                 float inx, float iny)
{
    OceanExp o;
    o.u = P.uo_x; o.v = P.uo_y; o.z = 0.0f;
    o.ux = o.uy = o.vx = o.vy = o.zx = o.zy = 0.0f;
    for (int m = 0; m < P.n_modes; m++) {
        const float *M = S.mode[m];
        float cs, sn;
        if (P.taylor) {
            float c0, s0;
            rot_small(fmaf(M[0], xf, M[1] * yf), c0, s0);
            const float2 C = S.Cm[ci][m];
            cs = C.x * c0 - C.y * s0;
            sn = C.y * c0 + C.x * s0;
        } else {
            const float cyc = S.Cm[ci][m].x + turn_x(P, m, xf, inx) + turn_y(P, m, yf, iny);
            sincospif(2.0f * cyc, &sn, &cs);
        }
        // mode m: u -= Au cos(th), v += Av cos(th), curl -= Az sin(th), th = kx X + ky Y + phi
        const float kx = M[2], ky = M[3];
        const float au = M[4], av = M[5], az = M[6];
        o.u -= au * cs;
        o.v += av * cs;
        o.z -= az * sn;
        const float aus = au * sn, avs = av * sn, azc = az * cs;
        o.ux += aus * kx;
        o.uy += aus * ky;
        o.vx -= avs * kx;
        o.vy -= avs * ky;
        o.zx -= azc * kx;
        o.zy -= azc * ky;
    }
    return o;
}

// The contact law (contact_force) rounded operation by operation: every place
// that calls it gets the same force for the same pair, whatever the compiler
// would contract around it.  RD: is d = d2 id rounded before the sums it goes
// into?  Cells of up to 256 floes take it unrounded, larger ones rounded, as
// the two always have: the motion of packed floes magnifies a last-bit change
// of a force a thousandfold within a few hundred steps (rounded in small
// cells too: rms 4e-5 after 200 steps), and nothing asks for one.
// P: the law's constants E, G, eta, mu, inv_h_ref.
template <bool RD, class Law>
__device__ __forceinline__ void contact_force32(float dx, float dy, float d2, float rl, float rj, float hl,
                                                float hj, float dux, float duy, float wl, float wj, const Law &P,
                                                float &gx, float &gy, float &ft, unsigned &deep)
{
    const float id = inv_sqrt(d2);
    const float nx = __fmul_rn(dx, id), ny = __fmul_rn(dy, id);
    const float S = __fadd_rn(rl, rj), D = __fsub_rn(rl, rj);
    const float d = __fmul_rn(d2, id);
    auto d_plus = [&](float x) { return RD ? __fadd_rn(d, x) : __fmaf_rn(d2, id, x); };
    const float delta = d_plus(-S);
    const float Q = __fmul_rn(d_plus(-D), d_plus(D));
    const float rmin = dmin(rl, rj);
    const float lens = __fmul_rn(root(__fmul_rn(__fmul_rn(-delta, d_plus(S)), Q)), id);
    const float c = Q <= 0.0f ? __fmul_rn(2.0f, rmin) : lens;
    const float chc = __fmul_rn(c, __fmul_rn(dmin(hl, hj), P.inv_h_ref));
    const float vn = __fmaf_rn(dux, nx, __fmul_rn(duy, ny));
    const float Fn = dmin(__fmul_rn(chc, __fmaf_rn(P.E, delta, __fmul_rn(P.eta, vn))), 0.0f);
    float vt = __fmaf_rn(duy, nx, -__fmul_rn(dux, ny));
    vt = __fmaf_rn(-wj, rj, vt);
    vt = __fmaf_rn(-wl, rl, vt);
    ft = __fmul_rn(__fmul_rn(chc, P.G), vt);
    const float cap = __fmul_rn(P.mu, -Fn);
    ft = dmax(dmin(ft, cap), -cap);
    gx = __fmaf_rn(Fn, nx, -__fmul_rn(ft, ny));
    gy = __fmaf_rn(Fn, ny, __fmul_rn(ft, nx));
    deep |= (delta < __fmul_rn(-0.5f, rmin)) ? 1u : 0u;
}

struct Law {
    float E, G, eta, mu, inv_h_ref;
};

// The contact forces on floe ps from its candidates e0 .. e1 (entries of V,
// or, all_pairs, floe numbers), found by a whole warp: a candidate per lane,
// added up in ascending order.  (x, y) force, z torque, w nonzero for a deep
// contact.
template <int RT, int K>
__device__ __forceinline__ float4 long_list_force(const RunSm<RT, K> &S, int cur, int ps, int e0, int e1, bool all_pairs,
                                               float sx, float sy, Law P)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint2 qs = S.buf[cur].Q[ps];
    const float4 as = S.buf[cur].A[ps];
    const float rs = S.buf[cur].R[ps];
    float fx = 0.0f, fy = 0.0f, tq = 0.0f;
    unsigned deep = 0;
    for (int e = e0; e < e1; e += 32) {
        const bool on = e + lane < e1;
        const int q = !on ? ps : (all_pairs ? e + lane : (int)S.V[e + lane]);
        const PairSep s = pair_sep(S.buf[cur].Q[q], qs.x, qs.y, sx, sy);
        const float rq = S.buf[cur].R[q];
        const bool touch = q != ps && pair_touch(s, rs, rq);
        float gx = 0.0f, gy = 0.0f, ft = 0.0f;
        if (touch) {
            const float4 aq = S.buf[cur].A[q];
            contact_force32<(RT > RUN_T)>(s.dx, s.dy, s.d2, rs, rq, as.w, aq.w, __fsub_rn(aq.x, as.x), __fsub_rn(aq.y, as.y), as.z, aq.z,
                          P, gx, gy, ft, deep);
        }
        for (unsigned b = __ballot_sync(FULL, touch); b != 0u; b &= b - 1u) {
            const int i = __ffs((int)b) - 1;
            fx = __fadd_rn(fx, __shfl_sync(FULL, gx, i));
            fy = __fadd_rn(fy, __shfl_sync(FULL, gy, i));
            tq = __fmaf_rn(rs, __shfl_sync(FULL, ft, i), tq);
        }
    }
    return make_float4(fx, fy, tq, __any_sync(FULL, deep != 0u) ? 1.0f : 0.0f);
}

template <int RT, int K>
__global__ void __launch_bounds__(RT, MS_RUN_K1_BLOCKS * RUN_T / RT)
k_cell_run32_block(DevState32 in, DevState32 out, Phys<float> P, StepCommon sc, const int4 *groups, int ngroups,
                   const int4 *items, int qslot, int nsteps, float skin_steps)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RunSm<RT, K> &S = *reinterpret_cast<RunSm<RT, K> *>(smem_raw);
    constexpr int NW = RT / 32;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned FULL = 0xffffffffu;
    const float dt = sc.k.dt;
    const float sx = sc.k.sx, sy = sc.k.sy;
    const float Lcmin = fminf(sc.k.Lx, sc.k.Ly);
    const int nc = sc.ncell;
    const int j0 = (int)sc.i_local;                     // steps of the interval done before this run
    const bool have_tgt = sc.couple && sc.ctrl->have_tgt;
    const bool win_on = sc.couple != 0;
    const bool ends_interval = sc.couple && (j0 + nsteps == sc.N0);
    const bool carry_in = win_on && j0 > 0;             // the run continues a previous one inside its interval
    const bool carry_out = win_on && !ends_interval;
    const float dtsx = sc.k.dtsx, dtsy = sc.k.dtsy;
    const long long ncar = sc.ncarry;
    const int nev = sc.N0 / sc.n_t;                     // gradual updates per interval

    // wind of steps [js0, js0 + WIND) of the run (FP64 turn, once per block
    // for runs of up to WIND steps)
    auto wind_table = [&](int js0) {
        if (t < WIND && js0 + t < nsteps) {
            float ua, va;
            wind_at(P, (double)(sc.ctrl->base + j0 + js0 + t) * sc.dt, ua, va);
            S.wind[t] = make_float2(ua, va);
        }
    };
    wind_table(0);
    if (t < P.n_modes) {
        float *M = S.mode[t];
        M[0] = P.ta[t]; M[1] = P.tb[t];
        M[2] = P.mKx[t]; M[3] = P.mKy[t];
        M[4] = P.mAu[t]; M[5] = P.mAv[t]; M[6] = P.mAz[t];
    }

    for (;;) {
        // ---- next group from the queue
        __syncthreads();
        if (t == 0) {
            int g = (int)atomicAdd(&sc.ctrl->gq[qslot][0], 1u);
            if (g >= ngroups) {
                __threadfence();
                const unsigned done = atomicAdd(&sc.ctrl->gq[qslot][1], 1u);
                if (done == gridDim.x - 1) {     // the last block out resets the queue for the next launch
                    sc.ctrl->gq[qslot][0] = 0u;
                    sc.ctrl->gq[qslot][1] = 0u;
                    __threadfence();
                }
            }
            S.item = g;
        }
        __syncthreads();
        const int gid = S.item;
        if (gid >= ngroups) return;

        // ---- the group's cells
        const int4 gd = groups[gid];          // first slot, cells, floes, bins (with one large slot per cell)
        if (t < 32) {                         // warp 0: a group has at most 32 cells
            int n = 0;
            if (t < gd.y) {
                const int4 id = items[gd.x + t];  // cell, first floe in the group, bins per side, bin base
                const int c = id.x;
                const int skip = sc.skip && sc.skip[c] ? 1 : 0;
                n = skip ? 0 : sc.off[c + 1] - sc.off[c];
                S.cc[t] = c;
                S.cskip[t] = skip;
                S.cn[t] = n;
                S.cnb[t] = id.z;
                S.cbb[t] = id.w;
                S.cgo[t] = sc.off[c];
            }
            // the group's floes packed cell after cell, closure cells holding
            // none (without a closure: the places the grouping gave them)
            int x = n;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(FULL, x, d);
                if (lane >= d) x += y;
            }
            if (t < gd.y) S.cfs[t] = x - n;
            if (t == 31) S.nfl = x;
            const unsigned sk = __ballot_sync(FULL, t < gd.y && sc.skip && sc.skip[S.cc[t]]);
            if (t == 0) S.allskip = __popc(sk) == gd.y;
        }
        if (t == 0) {
            S.ncg = gd.y;
            S.nbin = gd.w;
        }
        if (t < 3 * GCMAX) (&S.cflag[0][0])[t] = sc.fresh;
        __syncthreads();
        if (S.allskip) continue;              // every cell of the group takes the closure this interval
        const int ncg = S.ncg, nfl = S.nfl;
        for (int idx = t; idx < ncg * P.n_modes; idx += RT) {
            const int ci = idx / P.n_modes, m = idx - ci * P.n_modes;
            const int c = S.cc[ci];
            const float b = corner_phase(P, m, c % sc.g.nx, (c / sc.g.nx) % sc.g.nyr, sc.g.nx, sc.g.nyr, sc.k.inx,
                                         sc.k.iny);
            if (P.taylor) {
                float sn, cs;
                sincospif(2.0f * b, &sn, &cs);
                S.Cm[ci][m] = make_float2(cs, sn);
            } else {
                S.Cm[ci][m] = make_float2(b, 0.0f);
            }
        }
        // the window sums so far, added to in sequence and stored at the run's
        // end (the same additions however the interval is split into runs)
        if (t < ncg)
            for (int q = 0; q < NWIN; q++) S.cwin[t][q] = win_on ? sc.win[(size_t)q * nc + S.cc[t]] : 0.0;
        // per cell and gradual update of the interval (FP64, once): the
        // update's radius ratio; and, by the updates already applied, the
        // growth the radii can still take (r goes to r0 s at the last update
        // from r0 (1 + (s - 1) ev n_t/N0) after update ev) and the velocity the
        // remaining updates add (n_t/N0 of the target each)
        const int nevt = have_tgt && nev <= NEVT ? nev : 0;
        for (int idx = t; idx < ncg * (nevt + 1); idx += RT) {
            const int ci = idx / (nevt + 1), ev = idx - ci * (nevt + 1);
            const int c = S.cc[ci];
            const double s = sc.tgt[c];
            if (ev >= 1) S.rgev[ci][ev - 1] = (float)ramp_cell(sc, c, ev).g;
            float gr = 1.0f, dvr = 0.0f;
            if (nevt) {
                const double g = s / (1.0 + (s - 1.0) * ev / (double)nev);
                gr = g > 1.0 ? (float)(g * (1.0 + 1e-6)) : 1.0f;
                const double du = sc.tgt[nc + c], dv = sc.tgt[2 * nc + c];
                dvr = (float)(sqrt(du * du + dv * dv) * (nev - ev) / (double)nev);
            }
            S.cgrow[ci][ev] = gr;
            S.cdv[ci][ev] = dvr;
        }
        if (t == 0) {
            S.vsum[0] = S.vsum[1] = 0.0f;
            S.hz = fminf(skin_steps, 4.0f * (float)nsteps) * dt;   // a short run needs no wider skins
            S.nbuild = S.deep = 0;
            S.grp = make_int4(S.nfl, S.ncg, have_tgt, 0);
        }
        // gradual update of the run's first step, if it is one
        if (t < ncg) {
            const int kk = j0 + 1;
            float g = 1.0f, du = 0.0f, dv = 0.0f, dw = 0.0f;
            if (have_tgt && kk % sc.n_t == 0) {
                const RampCell rc = ramp_cell(sc, S.cc[t], kk / sc.n_t);
                g = (float)rc.g; du = (float)rc.du; dv = (float)rc.dv; dw = (float)rc.dw;
            }
            S.rg[0][t][0] = g; S.rg[0][t][1] = du; S.rg[0][t][2] = dv; S.rg[0][t][3] = dw;
        }

        // ---- this thread's floes: p = t + k RT in group order
        int ci[K], seg0[K], seg1[K];
        uint32_t xq[K], yq[K], x0[K], y0[K];
        float th[K], u[K], v[K], w[K], r[K];
        OceanExp oc[K];
        bool bad = false;
        // each slot's own constants, read once a step (D: kept out of the
        // registers, of which the step has 64)
        auto derived = [&](int k, float h) {
            const float mass = P.mass_c * r[k] * r[k] * h;
            const float I = P.inertia_f * mass * r[k] * r[k];
            S.D[t + k * RT].x = dt / mass;
            S.D[t + k * RT].y = dt / I;
        };
#pragma unroll
        for (int k = 0; k < K; k++) {
            const int s = t + k * RT;
            ci[k] = 0;
            seg0[k] = seg1[k] = 0;
            xq[k] = yq[k] = 0u;
            u[k] = v[k] = w[k] = 0.0f;
            r[k] = 1.0f;
            float h = 1.0f;
            th[k] = 0.0f;
            float su = 0.0f, sv = 0.0f, sfx = 0.0f, sfy = 0.0f, stz = 0.0f;
            if (s < nfl) {
                int c2 = 0;
                while (c2 + 1 < ncg && S.cfs[c2 + 1] <= s) c2++;
                ci[k] = c2;
                const int gi = S.cgo[c2] + (s - S.cfs[c2]), p = s;
                xq[k] = in.xq[gi]; yq[k] = in.yq[gi]; th[k] = in.th[gi];
                u[k] = in.u[gi]; v[k] = in.v[gi]; w[k] = in.w[gi]; r[k] = in.r[gi]; h = in.h[gi];
                S.buf[0].Q[p] = make_uint2(xq[k], yq[k]);
                S.buf[0].A[p] = make_float4(u[k], v[k], w[k], h);
                S.buf[0].R[p] = r[k];
            }
            x0[k] = xq[k];
            y0[k] = yq[k];
            if (carry_in && s < nfl) {
                const int gi = S.cgo[ci[k]] + (t + k * RT - S.cfs[ci[k]]);
                su = sc.carry_in[gi];
                sv = sc.carry_in[ncar + gi];
                sfx = sc.carry_in[2 * ncar + gi];
                sfy = sc.carry_in[3 * ncar + gi];
                stz = sc.carry_in[4 * ncar + gi];
                x0[k] = __float_as_uint(sc.carry_in[5 * ncar + gi]);
                y0[k] = __float_as_uint(sc.carry_in[6 * ncar + gi]);
            }
            S.W[s] = make_float4(su, sv, sfx, sfy);
            S.WT[s] = stz;
            S.D[s].z = 0.0f;
            S.D[s].w = h;
            derived(k, h);
        }
        // the ocean expansions are made in the step loop (one call site, so
        // every expansion rounds alike): at the first step about the places
        // above, later where a floe of the cell strays

        // ---- reduction of NV (<= NRED) per-floe values per cell, exact and
        // independent of where the cell's floes sit in the block: the
        // largest binary exponent of each (cell, column), then the values in
        // fixed point relative to it summed as integers (segments of a warp
        // by warp reductions, their heads into shared memory atomically);
        // head_sum converts a total back.  The columns are unrolled, so that their
        // chains overlap: a run of one step is a third reduction (393,216 floes in
        // cells of 6: 78 us, 70 so).  All threads call seg_partials; it begins and
        // ends with a barrier.
        auto seg_partials = [&](auto nv, auto &&value) {
            constexpr int NV = decltype(nv)::value;
            const int nfl = S.nfl;
            for (int i = t; i < NV * GCMAX; i += RT) {
                S.cexp[i / GCMAX][i % GCMAX] = FIX_NONE;
                S.csum[i / GCMAX][i % GCMAX] = 0ull;
            }
            __syncthreads();
            // a value counts if it is finite and nonzero (a non-finite state
            // is reported by the run's end check)
            auto counted = [&](int k, int q, bool valid) -> float {
                return fix_counted(valid ? value(k, q) : 0.0f);
            };
#pragma unroll
            for (int k = 0; k < K; k++) {
                const int p = t + k * RT;
                const bool valid = p < nfl;
                const int fs = valid ? S.cfs[ci[k]] : nfl;
                const int fe = valid ? S.cfs[ci[k]] + S.cn[ci[k]] : RT * K;
                const int wb = p & ~31;
                const int end_lane = min(fe, wb + 32) - wb;
                const int head = max(fs, wb);
                const bool whole = __all_sync(FULL, head == wb && end_lane == 32);
                const int longest = (int)__reduce_max_sync(FULL, (unsigned)(end_lane - (head - wb)));
#pragma unroll
                for (int q = 0; q < NV; q++) {
                    const float x = counted(k, q, valid);
                    const int e = seg_max(fix_exp(x), lane, end_lane, whole, longest);
                    if (p == head && e != FIX_NONE) atomicMax(&S.cexp[q][ci[k]], e);
                }
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < K; k++) {
                const int p = t + k * RT;
                const bool valid = p < nfl;
                const int fs = valid ? S.cfs[ci[k]] : nfl;
                const int fe = valid ? S.cfs[ci[k]] + S.cn[ci[k]] : RT * K;
                const int wb = p & ~31;
                const int end_lane = min(fe, wb + 32) - wb;
                const int head = max(fs, wb);
                const bool whole = __all_sync(FULL, head == wb && end_lane == 32);
                const int longest = (int)__reduce_max_sync(FULL, (unsigned)(end_lane - (head - wb)));
#pragma unroll
                for (int q = 0; q < NV; q++) {
                    const float x = counted(k, q, valid);
                    const long long iv = seg_sum(fix_val(x, S.cexp[q][ci[k]]), lane, end_lane, whole, longest);
                    if (p == head && iv != 0) atomicAdd(&S.csum[q][ci[k]], (unsigned long long)iv);
                }
            }
            __syncthreads();
        };
        auto head_sum = [&](int cell, int q) -> double {
            return fix_total((long long)S.csum[q][cell], S.cexp[q][cell]);
        };
        // ---- candidate lists from the positions in buffer b, before step kk.
        // The skins reach skin_steps steps ahead: twice that while floes have
        // less than one candidate on average (2.0M floes in cells of 6: two
        // builds per 100 steps instead of three, 2092 -> 2050 us), and half as
        // far, to an eighth, while the lists do not fit their room (true: call
        // again; testing every pair instead took 3.5 ms an interval on 115,200
        // floes where shorter skins take 0.5).
        int lists = 0;                    // 0: all short enough for a lane, 1: some longer, 2: they did not fit (every pair is tested)
        auto build = [&](int b, int kk) -> bool {
            const int nfl = S.nfl, ncg = S.ncg;
            const bool have_tgt = S.grp.z != 0;
            const int nev = sc.N0 / sc.n_t, nevt = have_tgt && nev <= NEVT ? nev : 0;
            // the floor of the skins: a quarter of the group's mean speed
            float vs = 0.0f;
#pragma unroll
            for (int k = 0; k < K; k++)
                if (t + k * RT < nfl) vs += sqrtf(u[k] * u[k] + v[k] * v[k]);
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) vs += __shfl_xor_sync(FULL, vs, d);
            for (int i = t; i <= S.nbin; i += RT) S.BS[i] = 0;
            if (have_tgt && !nevt && t < ncg) {   // more updates per interval than the table holds
                const int c = S.cc[t];
                const double s = sc.tgt[c];
                const int ev = (kk - 1) / sc.n_t;
                const double g = s / (1.0 + (s - 1.0) * ev / (double)nev);
                const double du = sc.tgt[nc + c], dv = sc.tgt[2 * nc + c];
                S.cgrow[t][0] = g > 1.0 ? (float)(g * (1.0 + 1e-6)) : 1.0f;
                S.cdv[t][0] = (float)(sqrt(du * du + dv * dv) * (nev - ev) / (double)nev);
            }
            const int vb = S.nbuild & 1;
            if (lane == 0) atomicAdd(&S.vsum[vb], vs);
            if (t == 0) {
                S.vsum[vb ^ 1] = 0.0f;    // for the next build
                S.nov = 0;
            }
            __syncthreads();
            // updates already applied (radius growth and velocity still to come)
            int evd = (kk - 1) / sc.n_t;
            if (!nevt) evd = 0;
            const float vfloor = 0.25f * S.vsum[vb] / (float)max(nfl, 1);
            const float hz = S.hz, horizon = fabsf(hz);
#pragma unroll
            for (int k = 0; k < K; k++) {
                const int p = t + k * RT;
                if (p < nfl) {
                    const int c2 = ci[k], nb = S.cnb[c2];
                    const float sp = sqrtf(u[k] * u[k] + v[k] * v[k]) + S.cdv[c2][evd];
                    const float skin = (1.5f * sp + vfloor) * horizon + 1.0e-3f * r[k];
                    S.D[t + k * RT].z = skin * skin;
                    const float reach = r[k] * S.cgrow[c2][evd] + skin;
                    S.RE[p] = reach;
                    const bool small = nb >= 3 && reach <= 0.5f * (Lcmin / (float)nb);
                    const int bn = S.cbb[c2] + (small ? (int)(__umulhi(yq[k], (unsigned)nb) * nb +
                                                               __umulhi(xq[k], (unsigned)nb))
                                                      : nb * nb);
                    S.BF[p] = (unsigned short)bn;
                    atomicAdd(&S.BS[bn], 1);
                    S.LC[p] = 0;
                }
            }
            __syncthreads();
            if (t == 0) S.nbuild++;
            block_scan_bins(S, S.nbin + 1);   // BS[nbin] = the group's floes
            int at[K];                        // the floe's place in bin order
#pragma unroll
            for (int k = 0; k < K; k++) {
                at[k] = 0;
                if (t + k * RT < nfl) {
                    at[k] = atomicAdd(&S.BC[S.BF[t + k * RT]], 1);
                    S.SF[at[k]] = (unsigned short)(t + k * RT);
                }
            }
            __syncthreads();
            // search: every pair from one side, its hit recorded on both
#pragma unroll
            for (int k = 0; k < K; k++) {
                const int p = t + k * RT;
                if (p >= nfl) continue;
                const int c2 = ci[k], nb = S.cnb[c2], bb = S.cbb[c2];
                const uint2 ql = make_uint2(xq[k], yq[k]);
                const float rl = S.RE[p];
                auto add = [&](int a, int q) {
                    const int slot = atomicAdd(&S.LC[a], 1);
                    if (slot < LMAX) {
                        S.L[slot][a] = (unsigned short)q;
                    } else {
                        const int o = atomicAdd(&S.nov, 1);
                        if (o < RunSm<RT, K>::OV) S.OVP[o] = ((unsigned)a << 16) | (unsigned)q;
                    }
                };
                const int lg0 = S.BS[bb + nb * nb], lg1 = S.BS[bb + nb * nb + 1];   // the cell's large floes
                const bool small = (int)S.BF[p] != bb + nb * nb;
                // small floe: the rest of its bin with the next one in x, the
                // three bins of the next row (of every two neighbouring bins
                // one has the other among these; bins side by side are one
                // range unless they wrap), then the large floes.  Large floe:
                // the half of the large ones that follows it in a ring (an even
                // number's opposite one from the first half).
                const int bx = (int)__umulhi(ql.x, (unsigned)nb), by = (int)__umulhi(ql.y, (unsigned)nb);
                const int row = bb + by * nb, nrow = bb + (by + 1 == nb ? 0 : by + 1) * nb;
                const bool wE = bx + 1 == nb, wW = bx == 0;
                const int m = lg1 - lg0, me = at[k] - lg0;
                const int half = (m - 1) / 2 + ((m & 1) == 0 && me < m / 2 ? 1 : 0);
#pragma unroll 1
                for (int part = 0; part < (small ? 5 : 2); part++) {
                    int i0 = 0, i1 = 0;
                    if (!small) {
                        i0 = part == 0 ? at[k] + 1 : lg0;
                        i1 = part == 0 ? min(at[k] + 1 + half, lg1) : lg0 + (me + 1 + half - m);
                    } else if (part == 0) {
                        i0 = at[k] + 1;
                        i1 = S.BS[row + bx + (wE ? 1 : 2)];
                    } else if (part == 1) {
                        i0 = S.BS[nrow + (wW ? 0 : bx - 1)];
                        i1 = S.BS[nrow + (wE ? nb : bx + 2)];
                    } else if (part == 4) {
                        i0 = lg0;
                        i1 = lg1;
                    } else if (wE) {
                        const int q = part == 2 ? row : nrow;
                        i0 = S.BS[q];
                        i1 = S.BS[q + 1];
                    } else if (wW && part == 2) {
                        i0 = S.BS[nrow + nb - 1];
                        i1 = S.BS[nrow + nb];
                    }
                    // up to 32 tests, then their hits: a warp's lanes hit at
                    // different tests and would else record them one by one
                    for (; i0 < i1; i0 += 32) {
                        unsigned hits = 0u;
                        const int e = min(i1 - i0, 32);
                        for (int i = 0; i < e; i++) {
                            const int q = S.SF[i0 + i];
                            const uint2 qq = S.buf[b].Q[q];
                            const float dx = (float)(int)(qq.x - ql.x) * sx, dy = (float)(int)(qq.y - ql.y) * sy;
                            const float Ssum = rl + S.RE[q];
                            if (fmaf(Ssum, Ssum, -(dx * dx + dy * dy)) > 0.0f) hits |= 1u << i;
                        }
                        for (; hits != 0u; hits &= hits - 1u) {
                            const int q = S.SF[i0 + __ffs((int)hits) - 1];
#pragma unroll 1
                            for (int side = 0; side < 2; side++) add(side ? q : p, side ? p : q);
                        }
                    }
                }
            }
            __syncthreads();
            // the lists one after another in thread order
            const int nov = S.nov;
            int n[K];
#pragma unroll
            for (int k = 0; k < K; k++) {
                n[k] = t + k * RT < nfl ? S.LC[t + k * RT] : 0;
                int x = n[k];
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int y = __shfl_up_sync(FULL, x, d);
                    if (lane >= d) x += y;
                }
                seg1[k] = x;
                if (lane == 31) S.wtot[k][warp] = x;
            }
            __syncthreads();
            int total = 0;
#pragma unroll
            for (int k = 0; k < K; k++) {
                int base = 0;
                for (int i = 0; i < NW; i++) {
                    if (i == warp) base = total;
                    total += S.wtot[k][i];
                }
                seg1[k] += base;
                seg0[k] = seg1[k] - n[k];
            }
            const bool all_pairs = nov > RunSm<RT, K>::OV || total > RunSm<RT, K>::PAIRS;
            const float skin0 = skin_steps * dt;
            const bool again = all_pairs && hz > 0.126f * skin0;
            if (t == 0) {
                if (again) S.hz = 0.5f * fminf(horizon, skin0);
                else if (all_pairs) S.hz = -skin0;      // shorter skins do not help: no more of it
                else if (total < nfl) S.hz = 2.0f * skin0;
                else if (total < 3 * nfl) S.hz = skin0;
                else S.hz = fminf(horizon, skin0);
            }
            if (again) return true;     // (the first barrier of the next call comes before S.hz is read)
            bool longer = false;
            // the lists before their sort, owner's lane << 10 | partner: in the
            // buffer that the coming step fills after the build
            unsigned short *U = reinterpret_cast<unsigned short *>(&S.buf[b ^ 1]);
            static_assert(sizeof(unsigned short) * RunSm<RT, K>::PAIRS <= sizeof(S.buf[0]), "unsorted lists");
            if (!all_pairs) {
#pragma unroll
                for (int k = 0; k < K; k++) {
                    const int m = min(n[k], LMAX);
                    for (int i = 0; i < m; i++)
                        U[seg0[k] + i] = (unsigned short)(lane << 10 | S.L[i][t + k * RT]);
                    if (n[k] > LMAX) S.ST[t + k * RT] = lane << 16 | (seg0[k] + LMAX);
                }
                __syncthreads();
                if (nov > 0) {
                    for (int i = t; i < nov; i += RT) {
                        const unsigned o = S.OVP[i];
                        const int c = atomicAdd(&S.ST[o >> 16], 1);
                        U[c & 0xffff] = (unsigned short)((c >> 16) << 10 | (int)(o & 0xffffu));
                    }
                    __syncthreads();
                }
                // each list in ascending floe order: an entry's place is its rank
#pragma unroll
                for (int k = 0; k < K; k++) {
                    const int wa = __shfl_sync(FULL, seg0[k], 0), wb = __shfl_sync(FULL, seg1[k], 31);
                    for (int e0 = wa; e0 < wb; e0 += 32) {
                        const int e = e0 + lane;
                        const int ent = e < wb ? (int)U[e] : 0;
                        const int s0 = __shfl_sync(FULL, seg0[k], ent >> 10), s1 = __shfl_sync(FULL, seg1[k], ent >> 10);
                        if (e < wb) {
                            int rank = s0;
                            for (int j = s0; j < s1; j++) rank += (int)U[j] < ent ? 1 : 0;
                            S.V[rank] = (unsigned short)(ent & 1023);
                        }
                    }
                }
                __syncwarp();
            } else {
                // a floe's candidates: its cell's floes, by number in the group
#pragma unroll
                for (int k = 0; k < K; k++) {
                    const bool valid = t + k * RT < nfl;
                    seg0[k] = valid ? S.cfs[ci[k]] : 0;
                    seg1[k] = valid ? seg0[k] + S.cn[ci[k]] : 0;
                }
            }
#pragma unroll
            for (int k = 0; k < K; k++) {
                S.B[t + k * RT] = make_uint2(xq[k], yq[k]);
                longer |= n[k] > LSER;
            }
            longer = __syncthreads_or(longer) != 0;   // and a barrier before a floe publishes over U
            lists = all_pairs ? 2 : (longer ? 1 : 0);
            return false;
        };

        // the first step's recentring follows the rule of every later step:
        // a cell whose floe strayed from its centre takes new ones
#pragma unroll
        for (int k = 0; k < K; k++)
            if (t + k * RT < nfl && ocean_stale(xq[k], yq[k], x0[k], y0[k], sx, sy, P.ocean_d2)) S.cflag[0][ci[k]] = 1;
        if (nsteps > WIND) wind_table(0);   // a previous group left a later table
        __syncthreads();
        bool need_build = true;
        int ph = (j0 + 1) % sc.n_t;                       // kk mod n_t
        int fl_cur = 0;                                   // the step's stray flags: js mod 3
        for (int js = 0; js < nsteps; js++) {
            // few values live across a step: what is cheap to read or to work out
            // again is, of the 64 registers the pair law needs most
            const int kk = j0 + js + 1;                   // step within the interval, 1-based
            const int4 grp = S.grp;
            const int cur = js & 1, nfl = grp.x, ncg = grp.y;
            const bool have_tgt = grp.z != 0, first = js == 0;
            const int fl_nxt = fl_cur == 2 ? 0 : fl_cur + 1, fl_old = 3 - fl_cur - fl_nxt;
            if (js > 0 && (js & (WIND - 1)) == 0) {
                __syncthreads();
                wind_table(js);
                __syncthreads();
            }
            const bool period_end = ph == 0;
            if (need_build)
                while (build(cur, kk)) {
                }
            const float2 wa = S.wind[js & (WIND - 1)];
            const bool ramp = have_tgt && period_end;
            const int rb = js & 1;
            ph = ph + 1 == sc.n_t ? 0 : ph + 1;           // next step's kk mod n_t
            // next step's gradual update, published by the step barrier below
            if (have_tgt && ph == 0 && t < ncg && js + 1 < nsteps) {
                const int ev = (kk + 1) / sc.n_t;
                if (sc.N0 / sc.n_t <= NEVT) {
                    const double f = (double)sc.n_t / (double)sc.N0;
                    const int c = S.cc[t];
                    S.rg[rb ^ 1][t][0] = S.rgev[t][ev - 1];
                    S.rg[rb ^ 1][t][1] = (float)(sc.tgt[nc + c] * f);
                    S.rg[rb ^ 1][t][2] = (float)(sc.tgt[2 * nc + c] * f);
                    S.rg[rb ^ 1][t][3] = (float)(sc.tgt[3 * nc + c] * f);
                } else {
                    const RampCell rc = ramp_cell(sc, S.cc[t], ev);
                    S.rg[rb ^ 1][t][0] = (float)rc.g;
                    S.rg[rb ^ 1][t][1] = (float)rc.du;
                    S.rg[rb ^ 1][t][2] = (float)rc.dv;
                    S.rg[rb ^ 1][t][3] = (float)rc.dw;
                }
            }
            if (t < ncg) S.cflag[fl_old][t] = sc.fresh;   // read at the last step, written at the next one's end
            bool far = false;
#pragma unroll
            for (int k = 0; k < K; k++) {
                const int p = t + k * RT;
                const bool valid = p < nfl;
                // the ocean expansion: every floe of a cell expands again about
                // its current position when one of them strayed at the last
                // step (a decision of the cell alone, whatever shares its
                // block); at the run's first step each floe about its centre
                // unless it strayed from it; at every step of a run that hands
                // its centres to none (sc.fresh)
                const bool recentre = valid && S.cflag[fl_cur][ci[k]] != 0;
                if (recentre || first) {
                    if (recentre) {
                        x0[k] = xq[k];
                        y0[k] = yq[k];
                    }
                    oc[k] = ocean_expand(P, S, ci[k], (float)x0[k] * INV2_32F, (float)y0[k] * INV2_32F, sc.k.inx,
                                         sc.k.iny);
                }
                // contacts, ascending partner order: a floe of up to LSER candidates
                // walks its own list, the warp takes the longer lists together, a
                // candidate per lane (the pair arithmetic is rounded operation by
                // operation, so both ways give the same forces)
                float fx = 0.0f, fy = 0.0f, tq = 0.0f;
                unsigned dflag = 0;
                const int cnt = seg1[k] - seg0[k];
                if (cnt <= LSER && lists < 2) {
                    const float hl = S.D[p].w;
                    for (int i = seg0[k]; i < seg1[k]; i++) {
                        const int q = S.V[i];
                        const PairSep s = pair_sep(S.buf[cur].Q[q], xq[k], yq[k], sx, sy);
                        const float rq = S.buf[cur].R[q];
                        if (!pair_touch(s, r[k], rq)) continue;
                        const float4 aq = S.buf[cur].A[q];
                        float gx, gy, ft;
                        contact_force32<(RT > RUN_T)>(s.dx, s.dy, s.d2, r[k], rq, hl, aq.w, __fsub_rn(aq.x, u[k]), __fsub_rn(aq.y, v[k]), w[k],
                                      aq.z, P, gx, gy, ft, dflag);
                        fx = __fadd_rn(fx, gx);
                        fy = __fadd_rn(fy, gy);
                        tq = __fmaf_rn(r[k], ft, tq);
                    }
                }
                for (unsigned longs = lists ? __ballot_sync(FULL, cnt > LSER || (lists == 2 && cnt > 1)) : 0u; longs != 0u;
                     longs &= longs - 1u) {
                    const int src = __ffs((int)longs) - 1;
                    const int e0 = __shfl_sync(FULL, seg0[k], src), e1 = __shfl_sync(FULL, seg1[k], src);
                    const float4 f = long_list_force(S, cur, (t & ~31) + k * RT + src, e0, e1, lists == 2, sx, sy,
                                                     Law{P.E, P.G, P.eta, P.mu, P.inv_h_ref});
                    if (lane == src) {
                        fx = f.x;
                        fy = f.y;
                        tq = f.z;
                        dflag = f.w != 0.0f;
                    }
                }
                if (!valid) continue;
                const float4 own = S.D[t + k * RT];
                if (dflag) atomicAdd(&S.deep, 1);
                // ocean and wind drag (Eq. 2.1c-d)
                const OceanExp &o = oc[k];
                const float ex = (float)(int)(xq[k] - x0[k]) * sx, ey = (float)(int)(yq[k] - y0[k]) * sy;
                const float uo = fmaf(o.ux, ex, fmaf(o.uy, ey, o.u));
                const float vo = fmaf(o.vx, ex, fmaf(o.vy, ey, o.v));
                const float zeta = fmaf(o.zx, ex, fmaf(o.zy, ey, o.z));
                const float r2 = r[k] * r[k];
                const float ao = P.drag_o * r2, aa = P.drag_a * r2, bo = ao * r2;
                const float du_o = uo - u[k], dv_o = vo - v[k];
                const float so = fast_norm(du_o, dv_o);
                const float au = wa.x - u[k], av = wa.y - v[k];
                const float sa = fast_norm(au, av);
                const float dwo = 0.5f * zeta - w[k];
                const float Fdx = ao * du_o * so + aa * au * sa;
                const float Fdy = ao * dv_o * so + aa * av * sa;
                const float Td = bo * dwo * fabsf(dwo);
                fx += Fdx; fy += Fdy; tq += Td;
                // forward Euler (Sec. 3.1), periodic wrap by fixed-point overflow
                xq[k] += (uint32_t)__float2int_rn(dtsx * u[k]);
                yq[k] += (uint32_t)__float2int_rn(dtsy * v[k]);
                th[k] += dt * w[k];
                u[k] += own.x * fx;
                v[k] += own.x * fy;
                w[k] += own.y * tq;
                if (ramp) {                   // gradual update (Eqs. 3.5-3.7)
                    const float *g4 = S.rg[rb][ci[k]];
                    r[k] *= g4[0];
                    u[k] += g4[1];
                    v[k] += g4[2];
                    w[k] += g4[3];
                    derived(k, own.w);
                }
                if (win_on) {
                    float4 sums = S.W[p];
                    sums.x += u[k];
                    sums.y += v[k];
                    sums.z += Fdx;
                    sums.w += Fdy;
                    S.W[p] = sums;
                    S.WT[p] += Td;
                }
                if (js == nsteps - 1) {       // the drag of the run's last step (moment columns 9-11): its constants are done with
                    S.D[p].x = Fdx;
                    S.D[p].y = Fdy;
                    S.D[p].z = Td;
                }
                S.buf[cur ^ 1].Q[p] = make_uint2(xq[k], yq[k]);
                S.buf[cur ^ 1].A[p] = make_float4(u[k], v[k], w[k], own.w);
                S.buf[cur ^ 1].R[p] = r[k];
                const uint2 qb = S.B[t + k * RT];
                const float bx = (float)(int)(xq[k] - qb.x) * sx, by = (float)(int)(yq[k] - qb.y) * sy;
                far |= bx * bx + by * by > own.z;
                if (ocean_stale(xq[k], yq[k], x0[k], y0[k], sx, sy, P.ocean_d2)) S.cflag[fl_nxt][ci[k]] = 1;
            }
            need_build = __syncthreads_or(far) != 0;
            fl_cur = fl_nxt;
        }
        // ---- the run's end: the cell moments of its last step (every column)
        // and, at the interval's end, the window sums of Algorithm 1, in one
        // exact reduction
        const int nfle = S.nfl, ncge = S.ncg;
        {
            float em[K], eI[K];
#pragma unroll
            for (int k = 0; k < K; k++) {
                em[k] = P.mass_c * r[k] * r[k] * S.D[t + k * RT].w;
                eI[k] = P.inertia_f * em[k] * r[k] * r[k];
            }
            auto val = [&](int k, int q) -> float {
                const float m = em[k], I = eI[k];
                switch (q) {
                case 0: return m;
                case 1: return m * u[k];
                case 2: return m * v[k];
                case 3: return I;
                case 4: return I * w[k];
                case 5: return 3.14159265358979323846f * r[k] * r[k];
                case 6: return m * u[k] * u[k];
                case 7: return m * v[k] * v[k];
                case 8: return S.D[t + k * RT].x;
                case 9: return S.D[t + k * RT].y;
                case 10: return S.D[t + k * RT].z;
                case 11: return m * S.W[t + k * RT].x;
                case 12: return m * S.W[t + k * RT].y;
                case 13: return S.W[t + k * RT].z;
                case 14: return S.W[t + k * RT].w;
                default: return S.WT[t + k * RT];
                }
            };
            if (ends_interval) seg_partials(std::integral_constant<int, 16>{}, val);
            else seg_partials(std::integral_constant<int, 11>{}, val);
            // moment columns 1-11 are reduction columns 0-10
            for (int i = t; i < 11 * ncge; i += RT) {
                const int cell = i / 11, q = i - 11 * cell;
                if (!S.cskip[cell]) sc.mom[(size_t)S.cc[cell] * NMOM + 1 + q] = head_sum(cell, q);
            }
            if (t < ncge && !S.cskip[t]) sc.mom[(size_t)S.cc[t] * NMOM] = (double)S.cn[t];
            if (ends_interval) {
                if (t < 5 * ncge) {
                    const int cell = t / 5, q = t - 5 * cell;     // window column
                    const double x = head_sum(cell, 11 + q);
                    if (q < 2) {
                        const double M = head_sum(cell, 0);
                        if (M > 0.0) S.cwin[cell][q] += x / M;
                    } else {
                        S.cwin[cell][q] += x;
                    }
                }
#pragma unroll
                for (int k = 0; k < K; k++) {
                    const float4 sums = S.W[t + k * RT];
                    bad |= !(isfinite(sums.x) && isfinite(sums.y) && isfinite(S.WT[t + k * RT]));
                }
            }
        }
        __syncthreads();
        if (win_on && t < ncge && !S.cskip[t]) {
            const int c = S.cc[t];
            for (int q = 0; q < NWIN; q++) sc.win[(size_t)q * nc + c] = S.cwin[t][q];
        }
        // ---- back to global memory
#pragma unroll
        for (int k = 0; k < K; k++) {
            const int p = t + k * RT;
            if (p >= nfle) continue;
            bad |= !(isfinite(u[k]) && isfinite(v[k]) && isfinite(w[k]));
            const int gi = S.cgo[ci[k]] + (t + k * RT - S.cfs[ci[k]]);
            out.xq[gi] = xq[k]; out.yq[gi] = yq[k]; out.th[gi] = th[k];
            out.u[gi] = u[k]; out.v[gi] = v[k]; out.w[gi] = w[k]; out.r[gi] = r[k];
            if (out.h != in.h) out.h[gi] = S.D[t + k * RT].w;
            if (carry_out) {
                const float4 sums = S.W[p];
                sc.carry_out[gi] = sums.x;
                sc.carry_out[ncar + gi] = sums.y;
                sc.carry_out[2 * ncar + gi] = sums.z;
                sc.carry_out[3 * ncar + gi] = sums.w;
                sc.carry_out[4 * ncar + gi] = S.WT[p];
                sc.carry_out[5 * ncar + gi] = __uint_as_float(x0[k]);
                sc.carry_out[6 * ncar + gi] = __uint_as_float(y0[k]);
            }
        }
        // an empty cell of the group: zero moments
        if (t < ncge && S.cn[t] == 0 && !S.cskip[t]) {
            double *mo = sc.mom + (size_t)S.cc[t] * NMOM;
            for (int q = 0; q < NMOM; q++) mo[q] = 0.0;
        }
        if (__syncthreads_or(bad) && t == 0) atomicOr(&sc.ctrl->err, ERR_NONFINITE);
        bad = false;
        if (t == 0 && S.deep) atomicAdd(&sc.ctrl->deep, (unsigned long long)S.deep);
    }
}

// Fold the floes' running window sums into the window: a block per cell,
// the masses of the current state, fixed-order sums; the sums are cleared
// (the expansion centres are kept: they stay valid wherever the floes are).
__global__ void __launch_bounds__(128) k_carry_flush(DevState32 s, StepCommon sc, float *carry, long long ncarry)
{
    __shared__ double red[6][128];
    const int c = blockIdx.x, t = threadIdx.x;
    const int o = sc.off[c], n = sc.off[c + 1] - o;
    double a[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int i = t; i < n; i += 128) {
        const long long gi = o + i;
        const float r = s.r[gi], h = s.h[gi];
        const double m = (double)r * (double)r * (double)h;   // rho_ice pi cancels in the mean
        a[0] += m;
        a[1] += m * carry[gi];
        a[2] += m * carry[ncarry + gi];
        a[3] += carry[2 * ncarry + gi];
        a[4] += carry[3 * ncarry + gi];
        a[5] += carry[4 * ncarry + gi];
        for (int q = 0; q < 5; q++) carry[q * ncarry + gi] = 0.0f;
    }
    for (int q = 0; q < 6; q++) red[q][t] = a[q];
    __syncthreads();
    for (int w = 64; w > 0; w >>= 1) {
        if (t < w)
            for (int q = 0; q < 6; q++) red[q][t] += red[q][t + w];
        __syncthreads();
    }
    if (t == 0) {
        const int nc = sc.ncell;
        if (red[0][0] > 0.0) {
            sc.win[c] += red[1][0] / red[0][0];
            sc.win[nc + c] += red[2][0] / red[0][0];
        }
        sc.win[2 * nc + c] += red[3][0];
        sc.win[3 * nc + c] += red[4][0];
        sc.win[4 * nc + c] += red[5][0];
    }
}

}  // namespace

cudaError_t launch_carry_flush(const DevState32 &s, const StepCommon &sc, float *carry, long long ncarry,
                               cudaStream_t st)
{
    if (sc.ncell <= 0 || !carry) return cudaSuccess;
    k_carry_flush<<<sc.ncell, 128, 0, st>>>(s, sc, carry, ncarry);
    return cudaGetLastError();
}

// The kernel of each class, by the floes its blocks hold in units of RUN_T:
// f(kernel, threads, shared memory).  A floe a thread and 64 registers in each,
// 1024 threads an SM: the step is a chain of latencies that warps hide.  With
// two floes a thread and half the warps the class of 256 takes 2415 us an
// interval instead of 2044 (2.0M floes in cells of 6), and with one block an SM
// (two floes a thread in the largest class) the larger classes 2860 instead of
// 2560 (2.0M floes, lognormal cells) and 980 instead of 890 (500,658 floes).
template <class F>
static auto with_class(int K, F &&f)
{
    if (K == 1) return f(k_cell_run32_block<RUN_T, 1>, RUN_T, sizeof(RunSm<RUN_T, 1>));
    if (K == 2) return f(k_cell_run32_block<2 * RUN_T, 1>, 2 * RUN_T, sizeof(RunSm<2 * RUN_T, 1>));
    return f(k_cell_run32_block<4 * RUN_T, 1>, 4 * RUN_T, sizeof(RunSm<4 * RUN_T, 1>));
}

size_t run_block_smem(int K)
{
    return with_class(K, [](auto, int, size_t sm) { return sm; });
}

cudaError_t run_block_prepare()
{
    for (int K : {1, 2, 4}) {
        const cudaError_t e = with_class(K, [](auto kern, int, size_t sm) {
            return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        });
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Persistent grid of one class: as many blocks as fit on the device at once
// (at most one per group).
static int run_block_grid(int K, int ngroups)
{
    // (made by the first caller; others wait for it)
    struct Most {
        int of[3];
        Most()
        {
            int dev = 0, nsm = 0;
            cudaGetDevice(&dev);
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
            for (int i = 0; i < 3; i++) {
                const int b = with_class(1 << i, [](auto kern, int threads, size_t sm) {
                    int n = 0;
                    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, sm);
                    return n;
                });
                of[i] = (b > 0 ? b : 1) * (nsm > 0 ? nsm : 1);
            }
        }
    };
    static const Most most;
    const int g = most.of[K == 1 ? 0 : (K == 2 ? 1 : 2)];
    return g < ngroups ? g : ngroups;
}

cudaError_t launch_run_block(int K, const DevState32 &in, const DevState32 &out, const Phys<float> &P,
                             const StepCommon &sc, const int4 *groups, int ngroups, const int4 *items, int qslot,
                             int nsteps, float skin_steps, cudaStream_t st)
{
    if (ngroups <= 0 || nsteps <= 0) return cudaSuccess;
    const int grid = run_block_grid(K, ngroups);
    with_class(K, [&](auto kern, int threads, size_t sm) {
        kern<<<grid, threads, sm, st>>>(in, out, P, sc, groups, ngroups, items, qslot, nsteps, skin_steps);
        return 0;
    });
    return cudaGetLastError();
}

}  // namespace msd
