// fcd_cross.cuh -- the 1/2 crossings of a column of nodes, found by several warps.
//
// The extents of Eq. 42 need, along a line of values that is 0 beyond both
// ends, the first step i -> i + 1 that rises through 1/2 and the last one that
// falls through it. A column is cut into runs of consecutive rows, one warp
// each (lane = column); every run keeps its end values and the steps inside it,
// and the runs are joined in row order. Only the primal values decide, so the
// derivative forms find the same steps and evaluate them afterwards.
#pragma once

namespace fcd {

struct RunCross {
    double v0, v1;    // first and last value of the run
    int first, last;  // rising and falling step (row of its lower end), -2: none
    int n;            // values seen

    __device__ __forceinline__ void clear() {
        v0 = v1 = 0.0;
        first = last = -2;
        n = 0;
    }
    // the step from value a at row i to value b at row i + 1
    __device__ __forceinline__ void step(int i, double a, double b) {
        if (a < 0.5 && b >= 0.5 && first == -2) first = i;
        if (a >= 0.5 && b < 0.5) last = i;
    }
    // the value at row y, the next of this run
    __device__ __forceinline__ void add(int y, double v) {
        if (n) step(y - 1, v1, v);
        else v0 = v;
        v1 = v;
        n++;
    }
    // the run r that starts at row y, which follows the rows joined so far
    // (this starts as the empty run: value 0 before row 0)
    __device__ __forceinline__ void join(int y, const RunCross &r) {
        if (!r.n) return;
        step(y - 1, v1, r.v0);
        if (first == -2) first = r.first;
        if (r.last != -2) last = r.last;
        v1 = r.v1;
        n += r.n;
    }
    // the step off the last of ny rows
    __device__ __forceinline__ void close(int ny) { step(ny - 1, v1, 0.0); }
    __device__ __forceinline__ bool found() const { return first != -2 && last != -2; }
};

// Length between the two steps, V the values along the line (0 beyond it):
// lo = i + (1/2 - a)/(b - a), hi = i + (a - 1/2)/(a - b).
template <typename V, typename F>
__device__ __forceinline__ V cross_extent(int first, int last, int n, F at) {
    auto v = [&](int i) { return i < 0 || i >= n ? V(0.0) : at(i); };
    const V a = v(first), b = v(first + 1), c = v(last), d = v(last + 1);
    return (double(last) + (c - 0.5) / (c - d)) - (double(first) + (0.5 - a) / (b - a));
}

// Launch of a kernel that gives 32 columns to a cluster of CH blocks of `runs`
// warps: two rows a warp or more, up to the portable limit of 8 blocks.
constexpr int COLUMN_CLUSTER = 8;
template <typename... KA, typename... A>
inline void launch_columns(void (*kernel)(KA...), int runs, int nx, int ny, cudaStream_t s, A... args) {
    int ch = (ny + 2 * runs - 1) / (2 * runs);
    ch = ch < 1 ? 1 : (ch > COLUMN_CLUSTER ? COLUMN_CLUSTER : ch);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((nx + 31) / 32, ch);
    cfg.blockDim = dim3(32, runs);
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 1;
    at.val.clusterDim.y = ch;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Fixed-order block reduction of Q values per thread (NTHR a power of two, at
// least a warp): op over the lanes of each warp, then over the warps. Every
// thread gets the results. Small blocks on purpose: a block-wide FP64 operation
// of 1024 threads takes about 450 cycles of this GPU's FP64 pipe.
template <int NTHR, int Q, typename V, typename F>
__device__ __forceinline__ void block_reduce(V (&v)[Q], F op) {
    constexpr int NW = NTHR / 32;
    static_assert(NW >= 1 && NW <= 32 && (NW & (NW - 1)) == 0, "whole warps, a power of two");
    __shared__ V sh[Q][NW];
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
#pragma unroll
    for (int q = 0; q < Q; q++) {
        for (int o = 16; o > 0; o >>= 1) v[q] = op(v[q], __shfl_down_sync(0xffffffffu, v[q], o));
        if (lane == 0) sh[q][w] = v[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q; q++)  // each quantity's second stage by one thread
        if (t == 32 * (q % NW)) {
            V r = sh[q][0];
            for (int i = 1; i < NW; i++) r = op(r, sh[q][i]);
            sh[q][0] = r;
        }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q; q++) v[q] = sh[q][0];
    __syncthreads();
}

// The order of doubles >= 0 is that of their bits: max and min on the integer
// pipe. (NaN sorts above infinity; the callers hand in values >= 0.)
__device__ __forceinline__ long long order_bits(double v) { return __double_as_longlong(v + 0.0); }

}  // namespace fcd
