// cell_run64.cu -- FP64 msDEM cell steps for a run of fine steps in one
// launch, the cell in shared memory for the whole run (cells of up to
// RUN64_MAX floes; larger ones take k_cell_step64_brute step by step).
//
// What bounds it: an SM issues an FP64 warp instruction only every 16 cycles
// or so, and a step is a chain of them (separation, force, drag, Euler, cell
// sums).  So the FP64 work per step is cut to what the method needs:
//  - a floe tests only its candidates, the floes that can touch it before
//    the next search, found by FP32 tests on 32-bit fixed-point positions
//    whose reach covers their rounding.  The tests of the candidates and the
//    contact law are the FP64 ones, the sum in ascending partner order, so
//    the forces are those of the loop over all pairs bit for bit.  A search
//    runs at the start of a run, after a gradual update (radii change) and
//    when a floe's path since the last one exceeds its skin; a floe with more
//    than LM candidates tests its whole cell.
//  - the modes' sines and cosines turn from their values at the cell's
//    centre by the angle to the floe, whose sine and cosine are Taylor sums
//    (remainder below 2^-54 over the cell), instead of a sincos per mode.
//  - the divisions by the cell side and by mass and inertia are per run or
//    per gradual update.
//  - the six sums a step needs (mass, momentum and drag of the cell, for the
//    window) go through one butterfly that halves the columns as it halves
//    the lanes: 9 FP64 additions a warp instead of 30.
// Measured on 16 cells of 16 floes: 58 us a step as launches of the
// all-pairs kernel, 12.6 us here.
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"

namespace msd {

namespace {

constexpr int LM = 16;        // candidates per floe
constexpr int WT64 = 32;      // steps per wind table

struct Sm64 {
    double *X[2], *Y[2], *U[2], *V[2], *W[2];   // by step buffer
    double *R, *H, *TH, *DM, *DI;               // radius, thickness, angle, dt / mass, dt / inertia
    uint2 *Q;                                   // search: fixed-point position
    float *RE, *SK, *PA;                        // search: reach; skin; path since
    unsigned short *L, *C;                      // candidates [LM][n], their number (LM + 1: test the whole cell)
};

__host__ __device__ constexpr size_t floe_bytes64() { return 8 * 15 + 8 + 4 * 3 + 2 * (LM + 1); }

__device__ __forceinline__ Sm64 carve64(unsigned char *p, int n)
{
    Sm64 s;
    double *d = reinterpret_cast<double *>(p);
    for (int b = 0; b < 2; b++) {
        s.X[b] = d; d += n;
        s.Y[b] = d; d += n;
        s.U[b] = d; d += n;
        s.V[b] = d; d += n;
        s.W[b] = d; d += n;
    }
    s.R = d; d += n;
    s.H = d; d += n;
    s.TH = d; d += n;
    s.DM = d; d += n;
    s.DI = d; d += n;
    s.Q = reinterpret_cast<uint2 *>(d);
    s.RE = reinterpret_cast<float *>(s.Q + n);
    s.SK = s.RE + n;
    s.PA = s.SK + n;
    s.L = reinterpret_cast<unsigned short *>(s.PA + n);
    s.C = s.L + (size_t)LM * n;
    return s;
}

// (-1)^(k/2) / k!
__host__ __device__ constexpr double taylor_coef(int k)
{
    double f = 1.0;
    for (int i = 2; i <= k; i++) f *= (double)i;
    return ((k / 2) & 1 ? -1.0 : 1.0) / f;
}

// sin and cos of |a| <= 0.25 (N = 6) or 1.7 (N = 11) by their Taylor series:
// the sine to a^(2N-1), the cosine to a^(2N)
template <int N>
__device__ __forceinline__ void taylor_sincos(double a, double &s, double &c)
{
    const double a2 = a * a;
    double ps = taylor_coef(2 * N - 1), pc = taylor_coef(2 * N);
#pragma unroll
    for (int k = N - 1; k >= 1; k--) {
        ps = fma(ps, a2, taylor_coef(2 * k - 1));
        pc = fma(pc, a2, taylor_coef(2 * k));
    }
    s = a * ps;
    c = fma(pc, a2, 1.0);
}

// Sum over the warp of 8 columns: lane l ends with the total of column
// 4 bit4(l) + 2 bit3(l) + bit2(l).
__device__ __forceinline__ double butterfly8(double (&v)[8], int lane)
{
    const unsigned FULL = 0xffffffffu;
#pragma unroll
    for (int w = 4; w >= 1; w >>= 1) {
        const int d = 4 * w;
        const bool up = (lane & d) != 0;
#pragma unroll
        for (int i = 0; i < w; i++) {
            const double send = up ? v[i] : v[i + w], keep = up ? v[i + w] : v[i];
            v[i] = keep + __shfl_xor_sync(FULL, send, d);
        }
    }
    double x = v[0];
    x += __shfl_xor_sync(FULL, x, 2);
    x += __shfl_xor_sync(FULL, x, 1);
    return x;
}

template <int T>
__global__ void __launch_bounds__(T)
k_cell_run64(DevState64 in, DevState64 out, Phys<double> P, StepCommon sc, int persistent, int nsteps, int turn_class)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int NWARP = T / 32;
    __shared__ double red[2][NWARP][8], red2[NWARP][8], Cc[MAXM], Sc[MAXM];
    __shared__ double2 wind[WT64];
    __shared__ double FB[NWARP][3][32];   // per warp: the contact forces of up to 32 pairs
    __shared__ int sh_item, sh_vmax;
    const unsigned FULL = 0xffffffffu;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const Sm64 S = carve64(smem, sc.max_n);
    const double dt = sc.dt, Lx = sc.g.Lcx, Ly = sc.g.Lcy, iLx = 1.0 / Lx, iLy = 1.0 / Ly;
    const float sx = (float)(Lx * (1.0 / 4294967296.0)), sy = (float)(Ly * (1.0 / 4294967296.0));
    const int nc = sc.ncell, j0 = (int)sc.i_local;
    const long long base = sc.ctrl->base;
    const bool have_tgt = sc.couple && sc.ctrl->have_tgt;
    unsigned long long deep = 0;
    bool bad = false;

    for (int item = persistent ? -1 : (int)blockIdx.x;;) {
        if (persistent) {
            __syncthreads();
            if (t == 0) {
                const int it = (int)atomicAdd(&sc.ctrl->queue[0], 1u);
                if (it >= nc) {
                    __threadfence();
                    if (atomicAdd(&sc.ctrl->queue[1], 1u) == gridDim.x - 1) {   // the last block out resets the queue
                        sc.ctrl->queue[0] = 0u;
                        sc.ctrl->queue[1] = 0u;
                        __threadfence();
                    }
                }
                sh_item = it;
            }
            __syncthreads();
            item = sh_item;
        }
        if (item >= nc) break;
        const int c = sc.order[item];
        const int o = sc.off[c], n = sc.off[c + 1] - o;
        const int ix = c % sc.g.nx, iy = (c / sc.g.nx) % sc.g.nyr;
        const double X0 = ix * Lx, Y0 = iy * Ly;
        auto derived = [&](int l) {
            const double m = P.mass_c * S.R[l] * S.R[l] * S.H[l];
            S.DM[l] = dt / m;
            S.DI[l] = dt / (P.inertia_f * m * S.R[l] * S.R[l]);
        };
        for (int k = t; k < n; k += T) {
            S.X[0][k] = in.x[o + k]; S.Y[0][k] = in.y[o + k]; S.U[0][k] = in.u[o + k]; S.V[0][k] = in.v[o + k];
            S.W[0][k] = in.w[o + k]; S.R[k] = in.r[o + k]; S.H[k] = in.h[o + k]; S.TH[k] = in.th[o + k];
            derived(k);
        }
        for (int m = t; m < P.n_modes; m += T)
            sincos(P.mKx[m] * (X0 + 0.5 * Lx) + P.mKy[m] * (Y0 + 0.5 * Ly) + P.mPh[m], &Sc[m], &Cc[m]);
        double win = 0.0;   // warp 0, lanes 1-5: the cell's window sums so far
        if (sc.couple && warp == 0 && lane >= 1 && lane <= NWIN) win = sc.win[(size_t)(lane - 1) * nc + c];
        __syncthreads();
        int cur = 0;
        bool need = true;
        for (int js = 0; js < nsteps; js++) {
            const int kk = j0 + js + 1;          // step within the interval, 1-based
            if ((js & (WT64 - 1)) == 0) {
                if (js > 0) __syncthreads();
                if (t < WT64 && js + t < nsteps) {
                    double ua, va;
                    wind_at(P, (double)(base + j0 + js + t) * sc.dt, ua, va);
                    wind[t] = make_double2(ua, va);
                }
                __syncthreads();
            }
            const double *X = S.X[cur], *Y = S.Y[cur], *U = S.U[cur], *V = S.V[cur], *W = S.W[cur];
            const bool last = js == nsteps - 1;
            const bool ramp = have_tgt && kk % sc.n_t == 0;
            if (need) {
                // each floe's reach to the next search: its radius, what it moves in
                // 24 steps at its speed (at least half the cell's largest), 0.2 %
                // of its radius and the rounding of the FP32 tests
                if (t == 0) sh_vmax = 0;
                __syncthreads();
                float vmax = 0.0f;
                for (int l = t; l < n; l += T) {
                    const float u = (float)U[l], v = (float)V[l];
                    vmax = fmaxf(vmax, sqrtf(u * u + v * v));
                }
                atomicMax(&sh_vmax, __float_as_int(vmax));   // not negative: ordered as integers
                __syncthreads();
                vmax = __int_as_float(sh_vmax);
                for (int l = t; l < n; l += T) {
                    S.Q[l] = make_uint2((uint32_t)(long long)rint(X[l] * iLx * 4294967296.0),
                                        (uint32_t)(long long)rint(Y[l] * iLy * 4294967296.0));
                    const float u = (float)U[l], v = (float)V[l], r = (float)S.R[l];
                    const float speed = sqrtf(u * u + v * v);
                    const float skin = 24.0f * (float)dt * fmaxf(speed, 0.5f * vmax) + 2.0e-3f * r;
                    S.SK[l] = skin;
                    S.PA[l] = 1.0001f * (float)dt * speed;   // this step's move
                    S.RE[l] = (r + skin) * 1.00001f + 4.0e-7f * fmaxf((float)Lx, (float)Ly);
                }
                __syncthreads();
                for (int l = t; l < n; l += T) {
                    const uint2 ql = S.Q[l];
                    const float rl = S.RE[l];
                    int k = 0;
                    for (int j = 0; j < n; j++) {
                        const uint2 qj = S.Q[j];
                        const float dx = (float)(int)(qj.x - ql.x) * sx, dy = (float)(int)(qj.y - ql.y) * sy;
                        const float reach = rl + S.RE[j];
                        // a comparison that NaN passes: a state that is no more finite tests everything
                        if (j != l && !(dx * dx + dy * dy >= reach * reach)) {
                            if (k < LM) S.L[k * sc.max_n + l] = (unsigned short)j;
                            k++;
                        }
                    }
                    S.C[l] = (unsigned short)min(k, LM + 1);
                }
                __syncwarp();   // the other lanes of the warp read these lists below
            }
            RampCell rc = {1.0, 0.0, 0.0, 0.0};
            if (ramp) rc = ramp_cell(sc, c, kk / sc.n_t);
            const double2 wa = wind[js & (WT64 - 1)];
            double acc[NMOM];
#pragma unroll
            for (int k = 0; k < NMOM; k++) acc[k] = 0.0;
            bool far = false;
            for (int l0 = 32 * warp; l0 < n; l0 += T) {
                const int l = l0 + lane;
                const bool valid = l < n;
                const int lv = valid ? l : l0;
                const double xl = X[lv], yl = Y[lv], ul = U[lv], vl = V[lv], wl = W[lv], rl = S.R[lv], hl = S.H[lv];
                double fx = 0.0, fy = 0.0, tq = 0.0;
                unsigned dp = 0;
                // each lane tests its floe's candidates; the touching pairs of the
                // warp then take the law a pair per lane, and each lane adds up its
                // own floe's forces in ascending partner order
                const bool all = S.C[lv] > LM;
                const int cnt = valid ? (all ? n : (int)S.C[lv]) : 0;
                const int most = (int)__reduce_max_sync(FULL, (unsigned)cnt);
                for (int b = 0; b < most; b += 32) {
                    auto partner = [&](int floe, bool whole, int i) { return whole ? b + i : (int)S.L[(b + i) * sc.max_n + floe]; };
                    auto sep = [&](double xa, double ya, int j, double &dx, double &dy) {
                        dx = X[j] - xa;
                        dy = Y[j] - ya;
                        dx -= Lx * rint(dx * iLx);
                        dy -= Ly * rint(dy * iLy);
                        return dx * dx + dy * dy;
                    };
                    unsigned hits = 0u;
                    const int e = min(32, cnt - b);
                    for (int i = 0; i < e; i++) {
                        const int j = partner(l, all, i);
                        double dx, dy;
                        const double d2 = sep(xl, yl, j, dx, dy), s = rl + S.R[j];
                        if (j != l && d2 > 0.0 && d2 < s * s) hits |= 1u << i;
                    }
                    int end = __popc(hits);                   // the lane's pairs are begin .. end of the warp's
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const int y = __shfl_up_sync(FULL, end, d);
                        if (lane >= d) end += y;
                    }
                    const int begin = end - __popc(hits), total = __shfl_sync(FULL, end, 31);
                    for (int c0 = 0; c0 < total; c0 += 32) {
                        const int p = min(c0 + lane, total - 1);
                        int src = 0;                          // the lane whose pair this is
#pragma unroll
                        for (int d = 16; d >= 1; d >>= 1)
                            if (__shfl_sync(FULL, end, src + d - 1) <= p) src += d;
                        unsigned h = __shfl_sync(FULL, hits, src);
                        for (int k = p - __shfl_sync(FULL, begin, src); k > 0; k--) h &= h - 1u;
                        const int a = l0 + src, j = partner(a, __shfl_sync(FULL, (int)all, src) != 0, __ffs((int)h) - 1);
                        double dx, dy, gx, gy, ft;
                        unsigned deep1 = 0;
                        const double d2 = sep(X[a], Y[a], j, dx, dy);
                        contact_force(dx, dy, d2, S.R[a], S.R[j], S.H[a], S.H[j], U[j] - U[a], V[j] - V[a], W[a], W[j], P, gx,
                                      gy, ft, deep1);
                        FB[warp][0][lane] = gx;
                        FB[warp][1][lane] = gy;
                        FB[warp][2][lane] = ft;
                        const unsigned D = __ballot_sync(FULL, deep1 != 0u);
                        __syncwarp();
                        for (int i = max(begin, c0); i < min(end, c0 + 32); i++) {
                            fx += FB[warp][0][i - c0];
                            fy += FB[warp][1][i - c0];
                            tq += rl * FB[warp][2][i - c0];
                            dp |= (D >> (i - c0)) & 1u;
                        }
                        __syncwarp();
                    }
                }
                if (!valid) continue;
                deep += dp;
                double uo = P.uo_x, vo = P.uo_y, zeta = 0.0;
                if (turn_class < 2) {
                    const double ax = xl - 0.5 * Lx, ay = yl - 0.5 * Ly;
                    for (int m = 0; m < P.n_modes; m++) {
                        double s, co;
                        const double a = P.mKx[m] * ax + P.mKy[m] * ay;
                        if (turn_class == 0) taylor_sincos<6>(a, s, co);
                        else taylor_sincos<11>(a, s, co);
                        const double cth = Cc[m] * co - Sc[m] * s, sth = Sc[m] * co + Cc[m] * s;
                        uo -= P.mAu[m] * cth;
                        vo += P.mAv[m] * cth;
                        zeta -= P.mAz[m] * sth;
                    }
                } else {
                    ocean_f64(P, X0 + xl, Y0 + yl, uo, vo, zeta);
                }
                double Fdx, Fdy, Td;
                drag_force(P, uo, vo, zeta, wa.x, wa.y, ul, vl, wl, rl, Fdx, Fdy, Td);
                fx += Fdx; fy += Fdy; tq += Td;
                double xn = xl + dt * ul;
                double yn = yl + dt * vl;
                S.TH[l] += dt * wl;
                double un = ul + S.DM[l] * fx;
                double vn = vl + S.DM[l] * fy;
                double wn = wl + S.DI[l] * tq;
                if (!(xn >= 0.0 && xn < Lx)) xn -= Lx * floor(xn / Lx);
                if (!(yn >= 0.0 && yn < Ly)) yn -= Ly * floor(yn / Ly);
                double rn = rl;
                if (ramp) {
                    rn = rl * rc.g;
                    un += rc.du;
                    vn += rc.dv;
                    wn += rc.dw;
                }
                bad |= !(isfinite(un) && isfinite(vn) && isfinite(wn));
                S.X[cur ^ 1][l] = xn;
                S.Y[cur ^ 1][l] = yn;
                S.U[cur ^ 1][l] = un;
                S.V[cur ^ 1][l] = vn;
                S.W[cur ^ 1][l] = wn;
                // the path since the search, rounded up, with the next step's move
                const float pu = (float)un, pv = (float)vn;
                const float path = S.PA[l] + 1.0001f * (float)dt * sqrtf(pu * pu + pv * pv);
                S.PA[l] = path;
                far |= !(path <= S.SK[l]);
                const double m = P.mass_c * rn * rn * hl;
                acc[1] += m;
                acc[2] += m * un;
                acc[3] += m * vn;
                acc[9] += Fdx;
                acc[10] += Fdy;
                acc[11] += Td;
                if (last) {
                    const double I = P.inertia_f * m * rn * rn;
                    acc[4] += I;
                    acc[5] += I * wn;
                    acc[6] += 3.14159265358979323846 * rn * rn;
                    acc[7] += m * un * un;
                    acc[8] += m * vn * vn;
                }
            }
            if (sc.couple || last) {
                double v8[8] = {acc[1], acc[2], acc[3], acc[9], acc[10], acc[11], 0.0, 0.0};
                const double x = butterfly8(v8, lane);
                if ((lane & 3) == 0) red[js & 1][warp][lane >> 2] = x;
            }
            if (last) {
                double v8[8] = {acc[4], acc[5], acc[6], acc[7], acc[8], 0.0, 0.0, 0.0};
                const double x = butterfly8(v8, lane);
                if ((lane & 3) == 0) red2[warp][lane >> 2] = x;
            }
            need = __syncthreads_or(far) != 0;
            if (ramp && !last) {
                for (int l = t; l < n; l += T) {
                    S.R[l] *= rc.g;
                    derived(l);
                }
                need = true;
                __syncthreads();
            }
            if (warp == 0 && (sc.couple || last)) {
                double s = 0.0;
                for (int w = 0; w < NWARP; w++) s += red[js & 1][w][lane & 7];
                const double M = __shfl_sync(0xffffffffu, s, 0);
                // lanes 1-5: momentum x, y over mass; drag x, y, torque
                if (sc.couple && lane >= 1 && lane <= NWIN) {
                    if (lane > 2) win += s;
                    else if (M > 0.0) win += s / M;
                }
                if (last) {
                    double *mo = sc.mom + (size_t)c * NMOM;
                    double s2 = 0.0;
                    for (int w = 0; w < NWARP; w++) s2 += red2[w][lane & 7];
                    if (lane == 0) mo[0] = (double)n;
                    if (lane < 3) mo[1 + lane] = s;
                    else if (lane < 6) mo[6 + lane] = s;
                    if (lane < 5) mo[4 + lane] = s2;
                }
            }
            cur ^= 1;
            if (last) {
                const bool wr = out.r != in.r;
                for (int l = t; l < n; l += T) {
                    out.x[o + l] = S.X[cur][l];
                    out.y[o + l] = S.Y[cur][l];
                    out.th[o + l] = S.TH[l];
                    out.u[o + l] = S.U[cur][l];
                    out.v[o + l] = S.V[cur][l];
                    out.w[o + l] = S.W[cur][l];
                    if (have_tgt || wr) out.r[o + l] = ramp ? S.R[l] * rc.g : S.R[l];
                }
                if (sc.couple && warp == 0 && lane >= 1 && lane <= NWIN) sc.win[(size_t)(lane - 1) * nc + c] = win;
            }
        }
        if (!persistent) break;
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&sc.ctrl->err, ERR_NONFINITE);
    if (deep) atomicAdd(&sc.ctrl->deep, deep);
}

}  // namespace

size_t run64_smem(int max_n) { return floe_bytes64() * (size_t)(max_n > 0 ? max_n : 1) + 16; }

cudaError_t launch_cell_run64(const DevState64 &in, const DevState64 &out, const Phys<double> &P,
                              const StepCommon &sc, const CellLaunch &cl, int nsteps, cudaStream_t st)
{
    const int grid = cl.persistent ? cl.grid : sc.ncell;
    if (grid <= 0 || nsteps <= 0) return cudaSuccess;
    // the largest angle any mode turns by from a cell's centre to its corner
    double turn = 0.0;
    for (int m = 0; m < P.n_modes; m++) {
        const double a = 0.5 * (fabs(P.mKx[m]) * sc.g.Lcx + fabs(P.mKy[m]) * sc.g.Lcy);
        turn = a > turn ? a : turn;
    }
    const int cls = turn <= 0.25 ? 0 : (turn <= 1.7 ? 1 : 2);
    const size_t sm = run64_smem(sc.max_n);
    switch (cl.threads) {
    case 64: k_cell_run64<64><<<grid, 64, sm, st>>>(in, out, P, sc, cl.persistent, nsteps, cls); break;
    case 128: k_cell_run64<128><<<grid, 128, sm, st>>>(in, out, P, sc, cl.persistent, nsteps, cls); break;
    case 256: k_cell_run64<256><<<grid, 256, sm, st>>>(in, out, P, sc, cl.persistent, nsteps, cls); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t run64_prepare()
{
    const void *kern[3] = {(const void *)k_cell_run64<64>, (const void *)k_cell_run64<128>,
                           (const void *)k_cell_run64<256>};
    for (const void *k : kern) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)run64_smem(RUN64_MAX));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace msd
