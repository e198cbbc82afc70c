// fcd_obs.cu -- observables of the coupled step (arXiv 2410.11129, Sec. 2.5,
// Eqs. 38 and 42): phase masses, indicator-weighted centroids, extents of the
// 1/2 level sets of the shell (phi_1 + phi_2) and the core (phi_1), and the
// breakup test (the core touching the carrier). FP64 throughout; reductions
// run in a fixed order (per column, then one block over the columns) so that
// repeated calls give identical bits.
#include <climits>

#include <cooperative_groups.h>

#include "fcd_cross.cuh"
#include "fcd_internal.cuh"

namespace fcd {

constexpr int COLS = OBS_COLS;  // records per column (planes of nx values): see obs_columns

template <int MODE>
struct StoreO { using type = float; };
template <>
struct StoreO<MODE_FP64> { using type = double; };

__device__ __forceinline__ double c01(double v) { return v < 0.0 ? 0.0 : (v > 1.0 ? 1.0 : v); }

// Core at a node with phi_1 >= 1/2 next to a carrier node (phi_3 >= 1/2)
// inside the channel; smallest y*nx + x wins.
__global__ void obs_touch(int nx, int ny, const double *phi1, const double *phi2, ObsOut *out,
                          int open) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= nx || y >= ny) return;
    if (c01(phi1[(long long)y * nx + x]) < 0.5) return;
    for (int a = 1; a < 9; a++) {
        const int yy = y + cy(a);
        if (yy < 0 || yy >= ny) continue;
        int xx = x + cx(a);
        if (open && (xx < 0 || xx >= nx)) continue;  // outside an open channel
        xx = xx < 0 ? nx - 1 : (xx >= nx ? 0 : xx);
        const long long m = (long long)yy * nx + xx;
        if (c01(1.0 - phi1[m] - phi2[m]) >= 0.5) {
            atomicMin(&out->brk_now, (unsigned long long)((long long)y * nx + x));
            return;
        }
    }
}

// Phase fields and per-column records in one pass: phi_1, phi_2 of every node
// (for obs_touch), and per column masses (3), sum so, sum si, sum y*so,
// sum y*si, vertical extents of so and si, centre-line values of so and si, and
// whether a value is not finite.
// A cluster takes 32 columns (lane = column, so the 18 population loads are
// coalesced) and cuts them into CH blocks x RUNS warps of consecutive rows. Each
// block joins its runs in row order, the first block then the blocks: the
// result does not depend on scheduling. Bound by FP64 arithmetic, of which an SM does about 2.2
// operations a clock: with one thread per column walking all the rows (13
// blocks on 1600 columns) this was about 430 of the 536 us of an observation
// of the 1600 x 200 FP32 channel, with one block per 32 columns 72 us, with the
// clusters 29 us (cold caches); the whole call 85 us.
constexpr int RUNS = 8;  // runs of rows per block (one warp each)
template <typename T>
__device__ __forceinline__ bool finite_value(T v) { return fabs(v) < T(1e300); }
template <>
__device__ __forceinline__ bool finite_value<float>(float v) { return fabsf(v) < INFINITY; }

template <typename T, int MODE>
__global__ void __launch_bounds__(32 * RUNS) obs_columns(Phys<T> P, const void *gv, double *phi1,
                                                         double *phi2, double *col, ObsOut *out) {
    using S = typename StoreO<MODE>::type;
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ double part[6][RUNS][32], bsum[6][32];
    __shared__ RunCross cross[2][RUNS][32], bcross[2][32];
    __shared__ int bad[32];
    const S *g = static_cast<const S *>(gv);
    const int nx = P.nx, ny = P.ny, lane = threadIdx.x, run = threadIdx.y;
    const int x = blockIdx.x * 32 + lane, CH = (int)cluster.num_blocks();
    const int rows = (ny + CH * RUNS - 1) / (CH * RUNS);  // per run
    const int y0 = (blockIdx.y * RUNS + run) * rows, y1 = min(ny, y0 + rows);
    if (run == 0) bad[lane] = 0;
    if (blockIdx.x == 0 && blockIdx.y == 0 && run == 0 && lane == 0) out->brk_now = ~0ull;  // obs_touch follows
    __syncthreads();
    double v[6] = {0, 0, 0, 0, 0, 0};
    RunCross cr[2];
    cr[0].clear();
    cr[1].clear();
    if (x < nx) {
        for (int y = y0; y < y1; y++) {
            const long long n = (long long)y * P.pitch + x, m = (long long)y * nx + x;
            T p1 = T(0), p2 = T(0);
#pragma unroll
            for (int a = 0; a < 9; a++) {
                p1 += T(g[a * P.ps + n]) - g_off<MODE, T>(a);
                p2 += T(g[(9 + a) * P.ps + n]) - g_off<MODE, T>(a);
            }
            const double d1 = double(p1), d2 = double(p2);
            phi1[m] = d1;
            phi2[m] = d2;
            if (!finite_value(p1) || !finite_value(p2)) bad[lane] = 1;
            const double i1 = double(clamp01(p1)), o = i1 + double(clamp01(p2));
            v[0] += d1;
            v[1] += d2;
            v[2] += o;
            v[3] += i1;
            v[4] += y * o;
            v[5] += y * i1;
            cr[0].add(y, o);
            cr[1].add(y, i1);
        }
    }
#pragma unroll
    for (int q = 0; q < 6; q++) part[q][run][lane] = v[q];
    cross[0][run][lane] = cr[0];
    cross[1][run][lane] = cr[1];
    __syncthreads();
    static_assert(RUNS == 8, "warps 0-5 take the sums, 6 and 7 the crossings");
    if (run < 6) {
        double s = 0;
#pragma unroll
        for (int r = 0; r < RUNS; r++) s += part[run][r][lane];
        bsum[run][lane] = s;
    } else {
        RunCross all;
        all.clear();
#pragma unroll
        for (int r = 0; r < RUNS; r++) all.join((blockIdx.y * RUNS + r) * rows, cross[run - 6][r][lane]);
        bcross[run - 6][lane] = all;
    }
    __threadfence();  // the phase fields are read back by the first block below
    cluster.sync();
    if (cluster.block_rank() == 0 && x < nx) {
        auto at = [&](int w, int y) {
            const long long m = (long long)y * nx + x;
            const double p1 = __ldcg(phi1 + m);
            return w ? c01(p1) : c01(p1) + c01(__ldcg(phi2 + m));
        };
        auto total = [&](int q) {
            double s = 0;
            for (int r = 0; r < CH; r++) s += *cluster.map_shared_rank(&bsum[q][lane], r);
            return s;
        };
        for (int task = run; task < COLS; task += RUNS) {
            double r = 0.0;
            if (task < 2) {
                r = total(task);
            } else if (task == 2) {  // phi_3 = 1 - phi_1 - phi_2
                r = ny - total(0) - total(1);
            } else if (task < 7) {
                r = total(task - 1);
            } else if (task < 9) {
                const int w = task - 7;
                RunCross all;
                all.clear();
                for (int q = 0; q < CH; q++) all.join(q * RUNS * rows, *cluster.map_shared_rank(&bcross[w][lane], q));
                all.close(ny);
                if (all.found()) r = cross_extent<double>(all.first, all.last, ny, [&](int y) { return at(w, y); });
            } else if (task < 11) {
                const int w = task - 9;
                r = (ny & 1) ? at(w, ny / 2) : 0.5 * (at(w, ny / 2 - 1) + at(w, ny / 2));
            } else {
                for (int q = 0; q < CH; q++)
                    if (*cluster.map_shared_rank(&bad[lane], q)) r = 1.0;
            }
            col[(long long)task * nx + x] = r;
        }
    }
    cluster.sync();  // the other blocks' shared memory is read until here
}

constexpr int FIN = 512;

// open: the frame starts at the inlet (no periodic seam to cut). pack: the
// result and the context's records gathered for the host (nullptr: none).
__global__ void __launch_bounds__(FIN) obs_final(int nx, const double *col, ObsOut *out, int open,
                                                 ObsTail tail) {
    const int t = threadIdx.x;
    auto add = [](double a, double b) { return a + b; };
    // masses, and whether any column holds a value that is not finite
    double ms[3] = {0, 0, 0};
    long long ends[1] = {LLONG_MAX};
    int flag[1] = {0};
    auto c = [&](int q, int x) { return col[(long long)q * nx + x]; };
#pragma unroll 4
    for (int x = t; x < nx; x += FIN) {
        for (int q = 0; q < 3; q++) ms[q] += c(q, x);
        const double so = c(3, x);
        if (so == so) ends[0] = min(ends[0], order_bits(so));
        flag[0] |= c(11, x) != 0.0;
    }
    auto least = [](auto a, auto b) { return min(a, b); };
    auto most = [](auto a, auto b) { return max(a, b); };
    block_reduce<FIN>(ms, add);
    block_reduce<FIN>(flag, most);
    // emptiest column (first of the minima): the seam for the periodic frame
    block_reduce<FIN>(ends, least);
    int xc[1] = {nx};
    for (int x = t; x < nx; x += FIN)
        if (order_bits(c(3, x)) == ends[0]) xc[0] = min(xc[0], x);
    block_reduce<FIN>(xc, least);
    const int xcut = open || xc[0] >= nx ? 0 : xc[0];
    double mo[6] = {0, 0, 0, 0, 0, 0};  // mass, x and y moments of the two indicators
    long long ly[2] = {0, 0};
    int first[2] = {INT_MAX, INT_MAX}, last[2] = {-3, -3};
#pragma unroll 4
    for (int x = t; x < nx; x += FIN) {
        const double xu = x >= xcut ? x : x + nx;
        for (int w = 0; w < 2; w++) {
            const double s = c(3 + w, x), l = c(7 + w, x);
            mo[3 * w] += s;
            mo[3 * w + 1] += xu * s;
            mo[3 * w + 2] += c(5 + w, x);
            if (l > 0.0) ly[w] = max(ly[w], order_bits(l));
        }
    }
    block_reduce<FIN>(mo, add);
    block_reduce<FIN>(ly, most);
    // centre-line crossings in the unwrapped frame j = 0..nx-1 (x = xcut + j), 0 beyond it:
    // the smallest upward and the largest downward one
    auto cl = [&](int w, int j) {
        if (j < 0 || j >= nx) return 0.0;
        const int x = xcut + j;
        return c(9 + w, x >= nx ? x - nx : x);
    };
#pragma unroll 4
    for (int i = t - 1; i < nx; i += FIN)
        for (int w = 0; w < 2; w++) {
            const double a = cl(w, i), b = cl(w, i + 1);
            if (a < 0.5 && b >= 0.5) first[w] = min(first[w], i);
            if (a >= 0.5 && b < 0.5) last[w] = max(last[w], i);
        }
    block_reduce<FIN>(first, least);
    block_reduce<FIN>(last, most);
    if (t != 0) return;
    ObsOut r;
    for (int q = 0; q < 3; q++) r.mass[q] = ms[q];
    double lx[2], xm[2], ym[2];
    for (int w = 0; w < 2; w++) {
        lx[w] = 0.0;
        if (first[w] != INT_MAX && last[w] != -3)
            lx[w] = cross_extent<double>(first[w], last[w], nx, [&](int j) { return cl(w, j); });
        xm[w] = mo[3 * w] > 0.0 ? fmod(mo[3 * w + 1] / mo[3 * w], (double)nx) : 0.0;
        ym[w] = mo[3 * w] > 0.0 ? mo[3 * w + 2] / mo[3 * w] : 0.0;
    }
    r.xc_shell = xm[0];
    r.yc_shell = ym[0];
    r.lx_o = lx[0];
    r.ly_o = __longlong_as_double(ly[0]);
    r.xc_core = xm[1];
    r.yc_core = ym[1];
    r.lx_i = lx[1];
    r.ly_i = __longlong_as_double(ly[1]);
    r.brk_now = out->brk_now;
    r.xcut = xcut;
    r.nonfinite = flag[0];
    *out = r;
    if (tail.pack) {
        tail.pack->o = r;
        tail.pack->brk = *tail.brk;
        tail.pack->unst = *tail.unst;
        tail.pack->ctl = *tail.ctl;
    }
}

template <typename T>
void launch_observe(int mode, const Phys<T> &P, const void *g, double *scratch, ObsOut *out,
                    cudaStream_t s, int open_x, ObsTail tail) {
    const long long N = (long long)P.nx * P.ny;
    double *phi1 = scratch, *phi2 = scratch + N, *col = scratch + 2 * N;
    if constexpr (sizeof(T) == 8) {
        launch_columns(obs_columns<T, MODE_FP64>, RUNS, P.nx, P.ny, s, P, g, phi1, phi2, col, out);
    } else {
        if (mode == MODE_FP32) launch_columns(obs_columns<T, MODE_FP32>, RUNS, P.nx, P.ny, s, P, g, phi1, phi2, col, out);
        else launch_columns(obs_columns<T, MODE_FP32_OFFSET>, RUNS, P.nx, P.ny, s, P, g, phi1, phi2, col, out);
    }
    dim3 b(32, 8), gr((P.nx + 31) / 32, (P.ny + 7) / 8);
    obs_touch<<<gr, b, 0, s>>>(P.nx, P.ny, phi1, phi2, out, open_x);
    obs_final<<<1, FIN, 0, s>>>(P.nx, col, out, open_x, tail);
}

size_t observe_scratch_doubles(int nx, int ny) { return observe_scratch_doubles_of(nx, ny); }

template void launch_observe<float>(int, const Phys<float> &, const void *, double *, ObsOut *,
                                    cudaStream_t, int, ObsTail);
template void launch_observe<double>(int, const Phys<double> &, const void *, double *,
                                     ObsOut *, cudaStream_t, int, ObsTail);

}  // namespace fcd
