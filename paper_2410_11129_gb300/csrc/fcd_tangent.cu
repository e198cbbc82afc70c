// fcd_tangent.cu -- kernels of the tangent-linear (forward-mode) step that are
// not shared with the plain step: the derivative planes of Eq. 32, Eq. 8 and
// the derivatives of the shell deformation T_o (Eq. 42) and of the core-carrier
// overlap sum_nodes phi_1 phi_3 (a smooth proxy of breakup, which happens when
// the core touches the carrier; unclamped fields, so that the sum is a
// polynomial of the state: the clamped product has a kink at every bulk node
// where phi sits at 0 or 1 up to round-off).
//
// Layout: every field plane set of the tangent context holds the primal value
// followed by NT tangent copies; copy c of plane q of an np-plane set sits
// (np * c + q) planes from the base.
#include <climits>

#include <cooperative_groups.h>

#include "fcd_cross.cuh"
#include "fcd_internal.cuh"

namespace fcd {

namespace {

__device__ __forceinline__ DualT ld_copies(const double *p, int q, int np, long long ps,
                                           long long n) {
    DualT r(p[q * ps + n]);
#pragma unroll
    for (int c = 0; c < NT; c++) r.d[c] = p[(np * (c + 1) + q) * ps + n];
    return r;
}

// phi_i = sum_a g^i_a and k = 1 / sum_i phi^_i / (1 + chi_i): derivative planes
// only (the primal planes come from the plain phase kernel).
__global__ void __launch_bounds__(256) tangent_phase_kernel(Phys<double> P, const double *g,
                                                            double *phi1, double *phi2, double *k) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const long long ps = P.ps, n = (long long)y * P.pitch + x;
    DualT p1(0.0), p2(0.0);
#pragma unroll
    for (int a = 0; a < 9; a++) {
        p1 += ld_copies(g, a, 18, ps, n);
        p2 += ld_copies(g, 9 + a, 18, ps, n);
    }
    const DualT kk = DualT(1.0) / (P.ik[0] * clamp01(p1) + P.ik[1] * clamp01(p2) +
                                   P.ik[2] * clamp01(DualT(1.0) - p1 - p2));
#pragma unroll
    for (int c = 0; c < NT; c++) {
        phi1[(c + 1) * ps + n] = p1.d[c];
        phi2[(c + 1) * ps + n] = p2.d[c];
        k[(c + 1) * ps + n] = kk.d[c];
    }
}

__device__ __forceinline__ DualT node_phi(const double *g, int base, long long ps, long long n) {
    DualT p(0.0);
#pragma unroll
    for (int a = 0; a < 9; a++) p += ld_copies(g, base + a, 18, ps, n);
    return p;
}

// Per column: the vertical 1/2-extent of the shell indicator phi^_1 + phi^_2,
// its centre-line value, and the column's part of the overlap; a cluster per 32
// columns, a run of rows per warp (see obs_columns). Bound by FP64 arithmetic
// (about 115 operations a node for the 90 planes of g): one block walking the
// columns of the 800 x 100 channel took 3.4 of the 3.5 ms of a tangent
// observation, one block per 32 columns 138 us, the clusters 63 us (cold caches).
constexpr int TRUNS = 8;
__global__ void __launch_bounds__(32 * TRUNS) tangent_obs_columns(int nx, int ny, int pitch, long long ps,
                                                                  const double *g, DualT *ext, DualT *cl,
                                                                  DualT *ovl) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ DualT part[TRUNS][32], bsum[32];
    __shared__ RunCross cross[TRUNS][32], bcross[32];
    const int lane = threadIdx.x, run = threadIdx.y, x = blockIdx.x * 32 + lane, CH = (int)cluster.num_blocks();
    const int rows = (ny + CH * TRUNS - 1) / (CH * TRUNS);
    const int y0 = (blockIdx.y * TRUNS + run) * rows, y1 = min(ny, y0 + rows);
    DualT o(0.0);
    RunCross cr;
    cr.clear();
    if (x < nx)
        for (int y = y0; y < y1; y++) {
            const long long n = (long long)y * pitch + x;
            const DualT p1 = node_phi(g, 0, ps, n), p2 = node_phi(g, 9, ps, n);
            o += p1 * (DualT(1.0) - p1 - p2);
            cr.add(y, clamp01(p1.v) + clamp01(p2.v));
        }
    part[run][lane] = o;
    cross[run][lane] = cr;
    __syncthreads();
    if (run == 0) {  // the block's runs in row order, then (below) the cluster's blocks
        RunCross all;
        all.clear();
        for (int r = 0; r < TRUNS; r++) all.join((blockIdx.y * TRUNS + r) * rows, cross[r][lane]);
        bcross[lane] = all;
    } else if (run == 1) {
        DualT s(0.0);
        for (int r = 0; r < TRUNS; r++) s += part[r][lane];
        bsum[lane] = s;
    }
    cluster.sync();
    if (cluster.block_rank() == 0 && x < nx) {
        auto at = [&](int y) {
            const long long n = (long long)y * pitch + x;
            return clamp01(node_phi(g, 0, ps, n)) + clamp01(node_phi(g, 9, ps, n));
        };
        if (run == 0) {
            RunCross all;
            all.clear();
            for (int q = 0; q < CH; q++) all.join(q * TRUNS * rows, *cluster.map_shared_rank(&bcross[lane], q));
            all.close(ny);
            ext[x] = all.found() ? cross_extent<DualT>(all.first, all.last, ny, at) : DualT(0.0);
        } else if (run == 1) {
            cl[x] = (ny & 1) ? at(ny / 2) : 0.5 * (at(ny / 2 - 1) + at(ny / 2));
        } else if (run == 2) {
            DualT s(0.0);
            for (int q = 0; q < CH; q++) s += *cluster.map_shared_rank(&bsum[lane], q);
            ovl[x] = s;
        }
    }
    cluster.sync();  // the other blocks' shared memory is read until here
}

// One block over the columns: l_y = the largest extent (first column among
// equal maxima), l_x from the centre-line crossings in the frame that starts at
// the emptiest column found by the plain observables, the overlap, and
// T_o = (l_y - l_x) / (l_y + l_x).
constexpr int TOB = 256;
__global__ void __launch_bounds__(TOB) tangent_obs_final(int nx, const DualT *ext, const DualT *cl,
                                                         const DualT *ovl, const ObsOut *prim, TanOut *out,
                                                         TanCtls ctls) {
    const int t = threadIdx.x, xcut = prim->xcut;
    auto clv = [&](int j) {
        const int x = xcut + j;
        return cl[x >= nx ? x - nx : x];
    };
    long long best[1] = {-1};  // extents are >= 0
    double tot[1 + NT] = {};
    int ij[2] = {INT_MAX, INT_MAX}, last[1] = {-3};  // first column of the maximum, rising step
    for (int x = t; x < nx; x += TOB) {
        if (ext[x].v >= 0.0) best[0] = max(best[0], order_bits(ext[x].v));
        tot[0] += ovl[x].v;
#pragma unroll
        for (int c = 0; c < NT; c++) tot[1 + c] += ovl[x].d[c];
    }
    auto least = [](int a, int b) { return min(a, b); };
    block_reduce<TOB>(best, [](long long a, long long b) { return max(a, b); });
    block_reduce<TOB>(tot, [](double a, double b) { return a + b; });
    for (int x = t; x < nx; x += TOB)
        if (order_bits(ext[x].v) == best[0]) ij[0] = min(ij[0], x);
    for (int i = t - 1; i < nx; i += TOB) {
        const double a = i < 0 ? 0.0 : clv(i).v, b = i + 1 < nx ? clv(i + 1).v : 0.0;
        if (a < 0.5 && b >= 0.5) ij[1] = min(ij[1], i);
        if (a >= 0.5 && b < 0.5) last[0] = max(last[0], i);
    }
    block_reduce<TOB>(ij, least);
    block_reduce<TOB>(last, [](int a, int b) { return max(a, b); });
    if (t != 0) return;
    const DualT ly = ij[0] < nx ? ext[ij[0]] : DualT(0.0);
    const DualT lx = ij[1] != INT_MAX && last[0] != -3 ? cross_extent<DualT>(ij[1], last[0], nx, clv) : DualT(0.0);
    const DualT To = (lx.v + ly.v) > 0.0 ? (ly - lx) / (ly + lx) : DualT(0.0);
    out->T_o = To.v;
    out->overlap = tot[0];
    out->lx = lx.v;
    out->ly = ly.v;
    out->nonconv = 0;
    for (int q = 0; q < NT; q++) {
        out->dT_o[q] = To.d[q];
        out->doverlap[q] = tot[1 + q];
        out->dlx[q] = lx.d[q];
        out->dly[q] = ly.d[q];
        if (ctls.c[q]) out->nonconv += ctls.c[q]->nonconv_count;
    }
}

}  // namespace

void launch_tangent_phase(const Phys<double> &P, const double *g, double *phi1, double *phi2,
                          double *k, cudaStream_t s) {
    dim3 b(32, 8), gr((P.nx + 31) / 32, (P.ny + 7) / 8);
    tangent_phase_kernel<<<gr, b, 0, s>>>(P, g, phi1, phi2, k);
}

size_t tangent_obs_scratch_bytes(int nx) { return 3ull * nx * sizeof(DualT); }

void launch_tangent_obs(const Phys<double> &P, const double *g, const ObsOut *prim, void *scratch,
                        TanOut *out, TanCtls ctls, cudaStream_t s) {
    DualT *ext = static_cast<DualT *>(scratch), *cl = ext + P.nx, *ovl = cl + P.nx;
    launch_columns(tangent_obs_columns, TRUNS, P.nx, P.ny, s, P.nx, P.ny, P.pitch, P.ps, g, ext, cl, ovl);
    tangent_obs_final<<<1, TOB, 0, s>>>(P.nx, ext, cl, ovl, prim, out, ctls);
}

}  // namespace fcd
