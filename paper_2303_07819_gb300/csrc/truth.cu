// truth.cu -- counting sorts on the device: the floes of a model grouped by
// cell (ms_init), and the truth DEM's floes binned by coarse cell for their
// moments (the truth steps themselves: truth_run.cu).
//
// Count -> scan -> scatter -> per-bin sort by floe index, so the bin contents
// and thus the summation order are deterministic.
#include <climits>

#include "common.cuh"
#include "upload.cuh"

namespace msd {

namespace {

constexpr int SCAN_T = 1024;

__global__ void k_scan_blocks(const int *in, int *out, int *bsum, int n)
{
    __shared__ int ws[32];
    const int i = blockIdx.x * SCAN_T + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int v = i < n ? in[i] : 0;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int t = ws[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        ws[lane] = t;
    }
    __syncthreads();
    const int incl = x + (warp > 0 ? ws[warp - 1] : 0);
    if (i < n) out[i] = incl - v;
    if (threadIdx.x == SCAN_T - 1) bsum[blockIdx.x] = incl;
}

// exclusive scan of the block sums, in place (nb <= SCAN_T)
__global__ void k_scan_top(int *bsum, int nb)
{
    __shared__ int ws[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int v = threadIdx.x < nb ? bsum[threadIdx.x] : 0;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int t = ws[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        ws[lane] = t;
    }
    __syncthreads();
    const int incl = x + (warp > 0 ? ws[warp - 1] : 0);
    if (threadIdx.x < nb) bsum[threadIdx.x] = incl - v;
}

__global__ void k_scan_add(int *out, const int *bsum, int n)
{
    const int i = blockIdx.x * SCAN_T + threadIdx.x;
    if (i < n) out[i] += bsum[blockIdx.x];
}

__global__ void k_set_int(int *p, int v) { *p = v; }

__global__ void k_scatter(const int *bin, const int *start, int *cursor, int *sorted, long long n)
{
    const long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= n) return;
    const int b = bin[l];
    sorted[start[b] + atomicAdd(&cursor[b], 1)] = (int)l;
}

// v[0..m) ascending, in place, by a warp: sorted runs of 1, 2, 4, ... merged in
// pairs, the first comparison of a merge mirrored, so that every comparison
// puts the smaller number lower and a run cut off at m needs no padding
// (Batcher's bitonic merge in its one-directional form).
__device__ void sort_long(int *v, int m)
{
    const int lane = threadIdx.x & 31;
    auto order = [&](long long i, long long j) {
        if (j >= m) return;
        const int a = v[i], b = v[j];
        if (a > b) {
            v[i] = b;
            v[j] = a;
        }
    };
    for (long long run = 1; run < m; run <<= 1) {
        const long long pairs = (m + 2 * run - 1) / (2 * run) * run;
        for (long long p = lane; p < pairs; p += 32) {
            const long long r = p & (run - 1), first = (p - r) * 2;
            order(first + r, first + 2 * run - 1 - r);
        }
        __syncwarp();
        for (long long d = run >> 1; d > 0; d >>= 1) {
            for (long long p = lane; p < pairs; p += 32) {
                const long long i = 2 * p - (p & (d - 1));
                order(i, i + d);
            }
            __syncwarp();
        }
    }
}

// Each bin's floe indices into ascending order, a warp per bin: every
// index's final place is its rank, the number of smaller indices in the bin
// (indices are distinct), so a lane ranks its entries against the bin's
// entries and all lanes write after all have read.  Bins of up to 32 floes
// rank from registers by shuffles; larger ones read the bin again per entry.
constexpr int SORT_WARPS = 8;

__global__ void __launch_bounds__(SORT_WARPS * 32) k_bin_sort(const int *start, int *sorted, int nbins)
{
    const int lane = threadIdx.x & 31;
    const int b = blockIdx.x * SORT_WARPS + (threadIdx.x >> 5);
    if (b >= nbins) return;
    const int s = start[b], m = start[b + 1] - s;
    if (m <= 1) return;
    int *bin = sorted + s;
    if (m <= 32) {
        const int key = lane < m ? bin[lane] : INT_MAX;
        int rank = 0;
        for (int i = 0; i < m; i++) rank += __shfl_sync(0xffffffffu, key, i) < key ? 1 : 0;
        __syncwarp();
        if (lane < m) bin[rank] = key;
        return;
    }
    // larger bins: at most 8 entries per lane held in registers until all
    // lanes have ranked theirs; up to 4096 floes, the most a cell starts with, a
    // serial insertion sort by lane 0 (the scatter leaves them nearly in order);
    // above that, floes of a run that piled up, or a diverged FP64 state's, all
    // of whose positions count as 0: merges by the warp, 0.1 s for 60,000 floes
    // where insertions could take the square of that
    if (m > 4096) {
        sort_long(bin, m);
        return;
    }
    if (m > 256) {
        if (lane == 0)
            for (int i = 1; i < m; i++) {
                const int key = bin[i];
                int j = i - 1;
                while (j >= 0 && bin[j] > key) {
                    bin[j + 1] = bin[j];
                    j--;
                }
                bin[j + 1] = key;
            }
        return;
    }
    int keys[8], ranks[8];
#pragma unroll
    for (int t = 0; t < 8; t++) {
        const int i = lane + 32 * t;
        keys[t] = i < m ? bin[i] : INT_MAX;
        ranks[t] = 0;
    }
    for (int i = 0; i < m; i++) {
        const int other = bin[i];
#pragma unroll
        for (int t = 0; t < 8; t++) ranks[t] += other < keys[t] ? 1 : 0;
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < 8; t++)
        if (lane + 32 * t < m) bin[ranks[t]] = keys[t];
}

// bin of a fixed-point coordinate: floor(frac * nb) exactly
__device__ __forceinline__ int fbin(uint32_t q, int nb) { return (int)(((unsigned long long)q * (unsigned)nb) >> 32); }

__device__ __forceinline__ int dbin(double x, double L, int nb)
{
    int b = (int)floor(x / (L / nb));
    return b < 0 ? 0 : (b > nb - 1 ? nb - 1 : b);
}

__global__ void k_bin32(const uint32_t *xq, const uint32_t *yq, TruthBins tb, long long n)
{
    const long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= n) return;
    const int b = fbin(yq[l], tb.nby) * tb.nbx + fbin(xq[l], tb.nbx);
    tb.bin[l] = b;
    atomicAdd(&tb.count[b], 1);
}

__global__ void k_bin64(const double *x, const double *y, double Lx, double Ly, TruthBins tb, long long n)
{
    const long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= n) return;
    const int b = dbin(y[l], Ly, tb.nby) * tb.nbx + dbin(x[l], Lx, tb.nbx);
    tb.bin[l] = b;
    atomicAdd(&tb.count[b], 1);
}

// --------------------------------------------------------- truth moments
// A warp per coarse cell: each lane sums every 32nd floe in ascending floe
// index in FP64, the lanes' sums add in a fixed tree (a thread per cell waits
// for each floe's loads in turn: 138 us on 1152 cells of 100 floes).
constexpr int MOM_WARPS = 4;

template <class R>
__global__ void __launch_bounds__(MOM_WARPS * 32)
k_truth_cell_moments(const R *u, const R *v, const R *w, const R *r, const R *h, const R *fd, long long n, double mass_c,
                     double inertia_f, const int *start, const int *sorted, int ncell, double *mom)
{
    const int lane = threadIdx.x & 31, c = blockIdx.x * MOM_WARPS + (threadIdx.x >> 5);
    if (c >= ncell) return;
    const int k0 = start[c], k1 = start[c + 1];
    double mo[NMOM];
    for (int k = 0; k < NMOM; k++) mo[k] = 0.0;
    for (int k = k0 + lane; k < k1; k += 32) {
        const int l = sorted[k];
        const double rl = r[l], hl = h[l], ul = u[l], vl = v[l], wl = w[l];
        const double m = mass_c * rl * rl * hl;
        const double I = inertia_f * m * rl * rl;
        mo[1] += m;
        mo[2] += m * ul;
        mo[3] += m * vl;
        mo[4] += I;
        mo[5] += I * wl;
        mo[6] += 3.14159265358979323846 * rl * rl;
        mo[7] += m * ul * ul;
        mo[8] += m * vl * vl;
        mo[9] += fd[l];
        mo[10] += fd[n + l];
        mo[11] += fd[2 * n + l];
    }
    double mine = (double)(k1 - k0);   // lane k ends with column k
#pragma unroll
    for (int k = 1; k < NMOM; k++) {
        double x = mo[k];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
        if (lane == k) mine = x;
    }
    if (lane < NMOM) mom[(size_t)c * NMOM + lane] = mine;
}

template <class BinF>
cudaError_t counting_sort(TruthBins &b, long long n, BinF binf, cudaStream_t st)
{
    const int nbins = b.nbins();
    cudaError_t e;
    if ((e = cudaMemsetAsync(b.count, 0, sizeof(int) * nbins, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(b.cursor, 0, sizeof(int) * nbins, st)) != cudaSuccess) return e;
    if (n > 0) binf();
    if ((e = bins_scan(b, nbins, st)) != cudaSuccess) return e;
    const int T = 256;
    if (n > 0) k_scatter<<<(unsigned)((n + T - 1) / T), T, 0, st>>>(b.bin, b.start, b.cursor, b.sorted, n);
    k_bin_sort<<<(nbins + SORT_WARPS - 1) / SORT_WARPS, SORT_WARPS * 32, 0, st>>>(b.start, b.sorted, nbins);
    return cudaGetLastError();
}

}  // namespace

// ---- the floes of a model grouped by cell (ms_init)

// exclusive scan of n ints (in place allowed): per-block scans, the block
// totals scanned the same way, then added back
static cudaError_t scan_exclusive(const int *in, int *out, long long n, int *tmp, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    const long long nb = (n + SCAN_T - 1) / SCAN_T;
    k_scan_blocks<<<(unsigned)nb, SCAN_T, 0, st>>>(in, out, tmp, (int)n);
    if (nb > 1) {
        const cudaError_t e = scan_exclusive(tmp, tmp, nb, tmp + nb, st);
        if (e != cudaSuccess) return e;
        k_scan_add<<<(unsigned)nb, SCAN_T, 0, st>>>(out, tmp, (int)n);
    }
    return cudaGetLastError();
}

long long sort_scan_ints(long long n)
{
    long long total = 1;
    while (n > 1) {
        n = (n + SCAN_T - 1) / SCAN_T;
        total += n;
    }
    return total + 1;
}

namespace {

constexpr int RANK_T = 256;
constexpr int RANK_MAX = 4096;   // the largest cell a model takes

// A block per cell: the cell's caller indices into ascending order, each
// entry placed at its rank (the number of smaller indices; they are
// distinct).  Cells above RANK_MAX floes are left as scattered (ms_init
// rejects them before this runs).
__global__ void __launch_bounds__(RANK_T) k_cell_rank_sort(const int *off, int *orig, int ncell)
{
    __shared__ int keys[RANK_MAX];
    const int c = blockIdx.x;
    if (c >= ncell) return;
    const int s = off[c], m = off[c + 1] - s;
    if (m <= 1 || m > RANK_MAX) return;
    for (int i = threadIdx.x; i < m; i += RANK_T) keys[i] = orig[s + i];
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += RANK_T) {
        const int key = keys[i];
        int rank = 0;
        for (int j = 0; j < m; j++) rank += keys[j] < key ? 1 : 0;
        orig[s + rank] = key;
    }
}

}  // namespace

cudaError_t sort_by_cell(const int *cell_of, const int *count, int *off, int *cursor, int *orig, int *tmp,
                         int ncell, long long n, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(cursor, 0, sizeof(int) * ncell, st);
    if (e == cudaSuccess) e = scan_exclusive(count, off, ncell, tmp, st);
    if (e != cudaSuccess) return e;
    k_set_int<<<1, 1, 0, st>>>(off + ncell, (int)n);
    const int T = 256;
    if (n > 0) k_scatter<<<(unsigned)((n + T - 1) / T), T, 0, st>>>(cell_of, off, cursor, orig, n);
    if (n > 0 && ncell > 0) k_cell_rank_sort<<<ncell, RANK_T, 0, st>>>(off, orig, ncell);
    return cudaGetLastError();
}

cudaError_t bins_scan(TruthBins &b, int nbins, cudaStream_t st)
{
    const int nb = (nbins + SCAN_T - 1) / SCAN_T;
    if (nb > SCAN_T) return cudaErrorInvalidValue;
    k_scan_blocks<<<nb, SCAN_T, 0, st>>>(b.count, b.start, b.scan_tmp, nbins);
    k_scan_top<<<1, SCAN_T, 0, st>>>(b.scan_tmp, nb);
    k_scan_add<<<nb, SCAN_T, 0, st>>>(b.start, b.scan_tmp, nbins);
    return cudaGetLastError();
}

cudaError_t launch_truth_moments32(const DevState32 &s, const Phys<float> &P, const TruthArgs &a,
                                   TruthBins &cells, double *mom, cudaStream_t st)
{
    const int T = 256;
    const unsigned G = (unsigned)((a.n + T - 1) / T);
    cudaError_t e = counting_sort(cells, a.n, [&] {
        k_bin32<<<G, T, 0, st>>>(s.xq, s.yq, cells, a.n);
    }, st);
    if (e != cudaSuccess) return e;
    const int nc = cells.nbx * cells.nby;
    k_truth_cell_moments<float><<<(nc + MOM_WARPS - 1) / MOM_WARPS, MOM_WARPS * 32, 0, st>>>(
        s.u, s.v, s.w, s.r, s.h, reinterpret_cast<const float *>(a.fd), a.n, (double)P.mass_c,
        (double)P.inertia_f, cells.start, cells.sorted, nc, mom);
    return cudaGetLastError();
}

cudaError_t launch_truth_moments64(const DevState64 &s, const Phys<double> &P, const TruthArgs &a,
                                   TruthBins &cells, double *mom, cudaStream_t st)
{
    const int T = 256;
    const unsigned G = (unsigned)((a.n + T - 1) / T);
    cudaError_t e = counting_sort(cells, a.n, [&] {
        k_bin64<<<G, T, 0, st>>>(s.x, s.y, a.g.Lx, a.g.Ly, cells, a.n);
    }, st);
    if (e != cudaSuccess) return e;
    const int nc = cells.nbx * cells.nby;
    k_truth_cell_moments<double><<<(nc + MOM_WARPS - 1) / MOM_WARPS, MOM_WARPS * 32, 0, st>>>(
        s.u, s.v, s.w, s.r, s.h, reinterpret_cast<const double *>(a.fd), a.n, P.mass_c, P.inertia_f,
        cells.start, cells.sorted, nc, mom);
    return cudaGetLastError();
}

// ----------------------------------------------- moments without allocating
// A variant of the per-cell moment binning above whose working memory (the
// counting sort's counts, starts, cursors and the sorted floe list) lives in
// one file-scope device array instead of buffers from cudaMalloc, for callers
// that must not allocate device memory while they run (see msdem.h).  Every
// call on a device reuses the same array: the counts and cursors are cleared
// at the start of each call, and two calls that run on the GPU at the same
// time corrupt each other.

namespace {

// cell of a caller's floe: each coordinate wrapped into [0, L) by
// X - L floor(X / L), then the half-open cell floor(X / (L / n)), clamped
// (rounding can put a wrapped X on L itself) -- the assignment ms_init makes
__device__ __forceinline__ int wrap_cell(double X, double L, int n)
{
    const double Xw = X - L * floor(X / L);
    int i = (int)floor(Xw / (L / n));
    return i < 0 ? 0 : (i > n - 1 ? n - 1 : i);
}

__global__ void k_bin_wrap64(const double *x, const double *y, double Lx, double Ly, TruthBins tb, long long n)
{
    const long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= n) return;
    const int b = wrap_cell(y[l], Ly, tb.nby) * tb.nbx + wrap_cell(x[l], Lx, tb.nbx);
    tb.bin[l] = b;
    atomicAdd(&tb.count[b], 1);
}

}  // namespace

}  // namespace msd

// Scratch of ms_cell_moments_noalloc: 3 * NA_CELLS + 1 + NA_SCAN ints for the
// cell counts, starts and cursors plus the scan's block sums, then 2 * NA_FLOES
// ints for each floe's cell and the floes sorted by cell (about 2.2 MB).
#define MS_NA_FLOES (1 << 18)
#define MS_NA_CELLS (1 << 14)
#define MS_NA_SCAN ((MS_NA_CELLS + 1 + 1023) / 1024)
static __device__ __align__(256) int ms_noalloc_scratch[3 * MS_NA_CELLS + 1 + MS_NA_SCAN + 2 * MS_NA_FLOES];

namespace msd {

long long noalloc_max_floes() { return MS_NA_FLOES; }
int noalloc_max_cells() { return MS_NA_CELLS; }

// Device address of the scratch array on the current device.  The address a
// host program sees for the symbol is only a host-side placeholder; the device
// address is looked up on every call, with the caller's device current, so a
// context that was torn down and created again (where the module may load at
// another address) never gets a stale pointer.
static cudaError_t noalloc_scratch(int **out)
{
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, ms_noalloc_scratch);
    if (e != cudaSuccess) return e;
    *out = reinterpret_cast<int *>(p);
    return cudaSuccess;
}

cudaError_t noalloc_cell_moments(const Geom &g, double mass_c, double inertia_f, long long n, const double *x,
                                 const double *y, const double *u, const double *v, const double *w,
                                 const double *r, const double *h, const double *fd, double *mom,
                                 cudaStream_t st)
{
    int *base = nullptr;
    cudaError_t e = noalloc_scratch(&base);
    if (e != cudaSuccess) return e;
    TruthBins b{};
    b.nbx = g.nx;
    b.nby = g.ny;
    const int nbins = g.nx * g.ny;
    b.count = base;
    b.start = b.count + MS_NA_CELLS;
    b.cursor = b.start + MS_NA_CELLS + 1;
    b.scan_tmp = b.cursor + MS_NA_CELLS;
    b.bin = b.scan_tmp + MS_NA_SCAN;
    b.sorted = b.bin + MS_NA_FLOES;
    b.nscan_blocks = (nbins + 1023) / 1024;
    k_set_int<<<1, 1, 0, st>>>(b.start + nbins, (int)n);
    const int T = 256;
    const unsigned G = (unsigned)((n + T - 1) / T);
    e = counting_sort(b, n, [&] {
        k_bin_wrap64<<<G, T, 0, st>>>(x, y, g.Lx, g.Ly, b, n);
    }, st);
    if (e != cudaSuccess) return e;
    k_truth_cell_moments<double><<<(nbins + MOM_WARPS - 1) / MOM_WARPS, MOM_WARPS * 32, 0, st>>>(u, v, w, r, h, fd, n, mass_c, inertia_f,
                                                                     b.start, b.sorted, nbins, mom);
    return cudaGetLastError();
}

}  // namespace msd
