// fcd_mg_solve.cuh -- one potential solve as one cooperative kernel.
//
// Solves to a tight tolerance (FP64; the FP32 hi + lo pair) run about ten
// multigrid cycles each, and on the lattices they are used on (10^4 to 10^5
// nodes) a cycle of separate kernels was bound by their boundaries: ten kernels,
// a while node and a switch node took 54 us per cycle on 200 x 40 and 72 us on
// 800 x 100, of which the arithmetic is a few microseconds. Here every block
// stays resident (cooperative launch, one block per SM at most), the phases of a
// cycle are separated by grid barriers of about 1.5 us, every block takes the
// same decisions from the same norm, and nothing returns to the host or to a
// graph node until the solve ends. Measured per step at tolerance 1e-10: 200 x 40
// 622 -> 245 us (12.0 -> 9.4 residuals), 800 x 100 827 -> 390 us (11.5 -> 9.9), both to
// errors no larger than before (stop_factor); the FP32 pair on 402 x 123 at 1e-5:
// step 79 -> 42 us. Bound by the chain of phases. Clock stamps of one block on
// 800 x 100: barriers with the wait for the slowest block a third, the grid-wide
// coarse levels a quarter, the residual (FP64: 57 cycles per operation of a warp)
// and the single-block levels a sixth each, the lattice sweeps a tenth; on 200 x 40:
// single-block levels 43%, barriers 23%, residual 18%, sweeps 14%. 6% of the issue
// slots are used. The FP64 form spills (128 registers of 512 threads: 192 bytes of
// stack, the second node's coefficients in the residual).
//
// A cycle is a defect correction: the lattice residual in the context's type
// (after which its norm decides) and its restriction; the coarse levels,
// grid-wide down to level lc, whose remaining levels one block keeps in shared
// memory for the whole solve (their coefficients are formed once); then the
// lattice's correction e = interpolated level-1 correction + two sweeps, in FP32
// like every correction, which the next residual adds to psi'. FP64 arithmetic
// (1/58 of FP32 here) is left in the residual alone, whose norm decides. The two
// sweeps are separate phases, so the second sees its neighbours' new values: a tile's
// second sweep against the same frozen ring gains nothing (numpy prototype of the
// 800 x 100 channel: 0.27 per cycle with one sweep, 0.29 with two frozen, 0.165 with
// two refreshed).
//
// Values that another block wrote in this kernel are read past the L1 cache
// (__ldcg). Every wait is bounded: a barrier that does not complete marks the
// context (Bound) and ends the kernel.
#pragma once

namespace fcd {

constexpr int SOLVE_THREADS = 512;             // one block per SM, up to 128 registers a thread
// Threads per lattice tile: 64 in a sweep (a 2 x 2 quad each, one node per
// colour), 128 in the residual (two nodes each: four warps, one per quarter of
// the SM, whose FP64 unit takes about 57 cycles for an operation of a warp).
constexpr int RT = 128;
constexpr int SOLVE_WORKERS = SOLVE_THREADS / QT, RESID_WORKERS = SOLVE_THREADS / RT;
constexpr int FVH = SOLVE_THREADS / 32;        // rows of a coarse-level tile (32 columns)
static_assert(SOLVE_WORKERS <= 15, "one named barrier per worker, barrier 0 is the block's");
// A cycle's correction falls short of the smooth errors by about a tenth, so it is
// scaled. numpy prototype, rate per cycle at 1, 1.04, 1.08 and 1.1: 800 x 100 0.172,
// 0.140, 0.126, 0.130; 200 x 40 0.163, 0.135, 0.126, 0.141; 400 x 122 0.209, 0.178,
// 0.138, 0.125; chi = 5 0.316, 0.292, 0.267, 0.241. Not for an odd number of rows,
// whose cells of three at the wall it overshoots (400 x 123: 0.210, at 1.05 0.295),
// nor where rows are not merged. Measured with solves that stop at the tolerance,
// 1 -> 1.08: residuals per solve 8.5 -> 7.6 on 800 x 100 at 1e-10 (485 -> 432 us per
// step) and 2.73 -> 2.44 at 1e-5 (180 -> 170), 9.0 -> 8.0 on 200 x 40 (270 -> 241): no
// slower at any tolerance from 1e-4 to 1e-12. Going straight to V-cycles (no two-grid
// cycles first) takes 457 us per step on 800 x 100 and 251 on 200 x 40.
constexpr TC OVER = TC(1.08);

// The FP32 residual and correction are in units of a power of two near the
// right-hand side's size (MgCtl::scale), which is the caller's: the seed of a
// gradient may be 1e-60, far below the FP32 range. A power of two changes no
// bits within that range. e: its exponent; 0 where there is no such size.
template <typename T>
struct Unit {
    int e;
    T value, inverse;
    __device__ __forceinline__ explicit Unit(double scale) {
        const int b = (__double2hiint(scale) >> 20) & 0x7ff;
        e = b == 0 || b == 0x7ff ? 0 : b - 1023;
        if (sizeof(T) == 4 && (e < -100 || e > 100)) e = 0;  // such a pair has left the FP32 range itself
        e = e < -1000 ? -1000 : (e > 1000 ? 1000 : e);
        value = T(__hiloint2double((1023 + e) << 20, 0));
        inverse = T(__hiloint2double((1023 - e) << 20, 0));
    }
    // v in this unit
    __device__ __forceinline__ TC of(float v) const { return v * (float)inverse; }
    // by its exponent, on the integer pipe: FP64 arithmetic bounds the residual
    // (a value that is not finite ends the solve at its norm)
    __device__ __forceinline__ TC of(double v) const {
        const int hi = __double2hiint(v), b = (hi >> 20) & 0x7ff, to = b == 0 ? 0 : min(max(b - e, 0), 0x7ff);
        return TC(__hiloint2double((hi & 0x800fffff) | (to << 20), __double2loint(v)));
    }
};

template <typename T>
struct SolveArgs {
    Level<T> L0;
    const Level<TC> *lv;
    int nl, lc;
    T H0c, H0s;
    MgCtl *ctl;
    Bound *bound;           // the context's: a barrier that gives up leaves its mark there
    int form_coef;          // FP64: form the node coefficients (else another solve of this k has)
    TC *r0, *eA, *eB, *k0;  // lattice planes of the correction: residual, e (two buffers), k
};

// Grid barrier of a cooperative launch; ctl->bar counts arrivals from the
// solve's reset on. False once a barrier has timed out.
__device__ __forceinline__ bool grid_barrier(MgCtl *c, Bound *bound, unsigned polls, unsigned &arrivals) {
    __shared__ int ok;
    arrivals += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&c->bar, 1u);
        unsigned seen = 0, spin = 0;
        bool good = true;
        while (true) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&c->bar) : "memory");
            if (seen >= arrivals) break;
            if (++spin >= polls || ((spin & 1023u) == 0 && *(volatile int *)&bound->stuck)) {
                good = false;
                atomicExch(&bound->stuck, 1);
                *(volatile int *)bound->told = 1;  // read after the stream has been synchronised
                break;
            }
        }
        __threadfence();
        ok = good ? 1 : 0;
    }
    __syncthreads();
    return ok != 0;
}

// The NTHR threads of one worker.
template <int NTHR>
__device__ __forceinline__ void worker_sync(int w) { asm volatile("bar.sync %0, %1;" ::"r"(w + 1), "n"(NTHR) : "memory"); }

// Patch of level-1 corrections that a tile and its ring interpolate from.
constexpr int PCX = SX / 2 + 2, PCY = SY / 2 + 2;

// Shared memory of one worker: the residual phase holds psi' (and k while the
// coefficients are formed), the sweeps the correction and k in FP32.
template <typename T, bool COMP>
struct ResidTile {
    T sp[SY + 2][SX + 2];
    T sl[COMP ? SY + 2 : 1][COMP ? SX + 2 : 1];
    T sk[SY + 2][SX + 2];
};
struct SweepTile {
    TC se[SY + 2][SX + 2], sk[SY + 2][SX + 2], ce[PCY][PCX];
    int y0[SY + 2], y1[SY + 2];  // rows of ce, -1: wall
    TC wy[SY + 2];
};

// f(q, ly, lx, node, inside) for this thread's entries of a tile with its ring,
// NTHR threads (warp w takes ring rows w, w + NTHR / 32, ..., lane l column l;
// the two last columns go to threads 0 .. 2 SY + 3); node: the lattice node,
// rows beyond the walls mirrored; inside: not such a row.
template <int NTHR>
__host__ __device__ constexpr int ring_rows() { return (SY + 2 + NTHR / 32 - 1) / (NTHR / 32); }
template <int NTHR, typename F>
__device__ __forceinline__ void ring_entries(int nx, int ny, int pitch, int x0, int y0, int tid, F f) {
    const int lane = tid & 31, warp = tid >> 5;
    constexpr int R = ring_rows<NTHR>();
    auto wrap = [&](int gx) {
        if (gx < 0) gx += nx;
        while (gx >= nx) gx -= nx;
        return gx;
    };
    const int gxa = wrap(x0 - 1 + lane), ex = SX + (tid & 1), gxe = wrap(x0 - 1 + ex);
#pragma unroll
    for (int q = 0; q <= R; q++) {
        const int ly = q < R ? warp + q * (NTHR / 32) : tid >> 1;
        if (q < R ? ly >= SY + 2 : tid >= 2 * (SY + 2)) continue;
        const int gy = y0 - 1 + ly, my = gy < 0 ? 0 : (gy >= ny ? ny - 1 : gy);
        f(q, ly, q < R ? lane : ex, (long long)my * pitch + (q < R ? gxa : gxe), gy == my);
    }
}

// One four-colour sweep of the correction on a 32 x 8 tile by 64 threads, a
// 2 x 2 quad each (see smooth0_tile): L e = r0, from the interpolated level-1
// correction (from == nullptr) or from `from`. Columns merge in pairs (nx is
// even), so column lx of the ring lies between columns lx / 2 and lx / 2 + 1 of
// the coarse patch, a quarter or three quarters of the way.
template <typename T>
__device__ __forceinline__ void sweep_tile(SweepTile &S, const SolveArgs<T> &A, const Level<TC> &L1, const TC *from,
                                           TC *to, TC over, int bx, int by, int w, int tid) {
    const int nx = A.L0.nx, ny = A.L0.ny, pitch = A.L0.pitch, x0 = bx * SX, y0 = by * SY;
    const int qx = 2 * (tid % (SX / 2)), qy = 2 * (tid / (SX / 2));
    TC kv[ring_rows<QT>() + 1], ev[ring_rows<QT>() + 1], rr[4];
    bool own[4];
    ring_entries<QT>(nx, ny, pitch, x0, y0, tid, [&](int q, int, int, long long n, bool) {
        kv[q] = __ldcg(A.k0 + n);
        ev[q] = from ? __ldcg(from + n) : TC(0);
    });
#pragma unroll
    for (int c = 0; c < 4; c++) {
        const int x = x0 + qx + (c & 1), y = y0 + qy + (c >> 1);
        own[c] = x < nx && y < ny;
        rr[c] = own[c] ? __ldcg(A.r0 + (long long)y * pitch + x) : TC(0);
    }
    if (!from) {
        const int I0 = x0 / 2 - 1, J0 = (L1.ny == ny ? y0 : y0 / 2) - 1;
        constexpr int NP = (PCX * PCY + QT - 1) / QT;
        TC cv[NP];
#pragma unroll
        for (int q = 0; q < NP; q++) {
            const int t = tid + q * QT, J = J0 + t / PCX;
            int I = I0 + t % PCX;
            I = I < 0 ? I + L1.nx : I;
            while (I >= L1.nx) I -= L1.nx;
            cv[q] = t < PCX * PCY && J >= 0 && J < L1.ny ? __ldcg(L1.e + (long long)J * L1.pitch + I) : TC(0);
        }
        if (tid < SY + 2) {
            const int gy = y0 - 1 + tid;
            const bool in = gy >= 0 && gy < ny;
            const int a = in ? A.L0.py0[gy] : -1, b = in ? A.L0.py1[gy] : -1;
            S.y0[tid] = a < 0 ? -1 : a - J0;
            S.y1[tid] = b < 0 ? -1 : b - J0;
            S.wy[tid] = in ? TC(A.L0.pwy[gy]) : TC(0);
        }
#pragma unroll
        for (int q = 0; q < NP; q++)
            if (tid + q * QT < PCX * PCY) (&S.ce[0][0])[tid + q * QT] = cv[q];
        worker_sync<QT>(w);
    }
    ring_entries<QT>(nx, ny, pitch, x0, y0, tid, [&](int q, int ly, int lx, long long, bool) {
        if (!from) {
            const int i = lx >> 1, ja = S.y0[ly], jb = S.y1[ly];
            const TC wx = (lx & 1) ? TC(0.75) : TC(0.25);
            const TC va = ja >= 0 ? S.ce[ja][i] + wx * (S.ce[ja][i + 1] - S.ce[ja][i]) : TC(0);
            const TC vb = jb >= 0 ? S.ce[jb][i] + wx * (S.ce[jb][i + 1] - S.ce[jb][i]) : TC(0);
            ev[q] = va + S.wy[ly] * (vb - va);
        }
        S.se[ly][lx] = ev[q];
        S.sk[ly][lx] = kv[q];
    });
    worker_sync<QT>(w);
    Node9<TC> nd[4];
    TC inv[4];
#pragma unroll
    for (int c = 0; c < 4; c++) {
        const int lx = qx + (c & 1) + 1, ly = qy + (c >> 1) + 1, y = y0 + ly - 1;
        auto kat = [&](int dx, int dy) { return S.sk[ly + dy][lx + dx]; };
        nd[c] = node9<TC, false>(kat, y, ny, TC(0), TC(0));
        if (y == 0) nd[c].diag += nd[c].c[4];  // e(ghost) = -e(node)
        if (y == ny - 1) nd[c].diag += nd[c].c[2];
        inv[c] = __fdividef(TC(1), nd[c].diag);
    }
#pragma unroll
    for (int c = 0; c < 4; c++) {
        const int lx = qx + (c & 1) + 1, ly = qy + (c >> 1) + 1, y = y0 + ly - 1;
        auto pat = [&](int dx, int dy) { return S.se[ly + dy][lx + dx]; };
        if (own[c]) {
            const TC v = (off9<TC, true>(nd[c], pat, y, ny) - rr[c]) * inv[c];
            S.se[ly][lx] = v;
            to[(long long)y * pitch + x0 + lx - 1] = over * v;
        }
        worker_sync<QT>(w);  // the last one: the tile's shared memory is reused
    }
}

// The order of values >= 0 is that of their bits, which the integer pipe
// compares (an FP64 operation of a warp takes about 14 cycles on this GPU); NaN
// sorts above infinity.
__device__ __forceinline__ long long max_bits(float v) { return (long long)__float_as_uint(fabsf(v)); }
__device__ __forceinline__ long long max_bits(double v) { return __double_as_longlong(v) & 0x7fffffffffffffffll; }
__device__ __forceinline__ double max_value(long long b, float) { return (double)__uint_as_float((unsigned)b); }
__device__ __forceinline__ double max_value(long long b, double) { return __longlong_as_double(b); }

// sum of c_a * psi~_a as off9, in two chains (FP64 latency)
template <typename T, typename PF>
__device__ __forceinline__ T off9_two(const Node9<T> &n, PF pat, int y, int ny) {
    T s[2] = {T(0), T(0)};
#pragma unroll
    for (int a = 1; a < 9; a++) {
        const int yy = y + cy(a);
        const bool ghost = cy(a) != 0 && (yy < 0 || yy >= ny);
        if (ghost && cx(a) == 0) continue;
        const T v = pat(cx(a), ghost ? 0 : cy(a));
        s[a & 1] += n.c[a] * (ghost ? -v : v);
    }
    return s[0] + s[1];
}

// psi' of a tile (plus the correction e, in units of `unit`, where there is one: written to psi_new),
// its residual (to r0) and the residual summed onto the tile's level-1 cells;
// returns the thread's max |r| (max_bits). A thread takes two neighbouring nodes
// of a row, and the two rows of a cell sit 16 lanes apart. first: the solve's
// first residual, which also forms what depends on k alone: the FP32 copy, the
// cells' mean, and (form) the FP64 node coefficients. An odd last row belongs to
// the cell below it: it is the ring's top row then, and a wall row, whose upper
// neighbours are ghosts.
template <typename T, bool COMP>
__device__ __forceinline__ long long resid_tile(ResidTile<T, COMP> &S, const SolveArgs<T> &A, const Level<TC> &L1,
                                                const T *psi, T *psi_new, const TC *e, const Unit<T> &unit, bool first,
                                                int bx, int by, int w, int tid) {
    const Level<T> &L0 = A.L0;
    const int nx = L0.nx, ny = L0.ny, pitch = L0.pitch, x0 = bx * SX, y0 = by * SY;
    const long long ps = (long long)pitch * ny;
    constexpr bool PLANES = keeps_coef<T>();
    const bool form = PLANES && first && A.form_coef;
    const bool load_k = !PLANES || first;
    static_assert(RT == (SX / 2) * SY, "two nodes per thread");
    const int ia = x0 + 2 * (tid % (SX / 2)), j0 = y0 + tid / (SX / 2);  // nx is even
    const bool merged = L1.ny != ny;                                     // not for ny <= 3
    const bool tail = merged && (ny & 1);                                // the last cell has three rows
    const bool live = ia < nx && j0 < ny - (tail ? 1 : 0);               // its last row: see below
    const bool third = live && tail && j0 == ny - 2;                     // this thread also takes row ny - 1
    auto coef = [&](Node9<T> &nd, int i, int j) {
        const long long n = (long long)j * pitch + i;
#pragma unroll
        for (int a = 1; a < 9; a++) nd.c[a] = __ldcg(L0.coef + (a - 1) * ps + n);
        nd.diag = __ldcg(L0.coef + 8 * ps + n);
        nd.b = L0.rhs ? L0.rhs[n] : __ldcg(L0.coef + 9 * ps + n);
    };
    Node9<T> pre[PLANES ? 2 : 1];
    if constexpr (PLANES) {
        if (!form && live) {
            coef(pre[0], ia, j0);
            coef(pre[1], ia + 1, j0);
        }
    }
    {
        constexpr int R = ring_rows<RT>() + 1;
        T pv[R], lv[COMP ? R : 1], kv[R];
        TC ev[R];
        ring_entries<RT>(nx, ny, pitch, x0, y0, tid, [&](int q, int, int, long long n, bool) {
            pv[q] = __ldcg(psi + n);
            if constexpr (COMP) lv[q] = __ldcg(psi + ps + n);
            ev[q] = e ? __ldcg(e + n) : TC(0);
            kv[q] = load_k ? L0.k[n] : T(0);
        });
        ring_entries<RT>(nx, ny, pitch, x0, y0, tid, [&](int q, int ly, int lx, long long n, bool inside) {
            if (e) {
                if constexpr (COMP) comp_add(pv[q], lv[q], ev[q] * unit.value);
                else pv[q] = fma(T(ev[q]), unit.value, pv[q]);
            }
            S.sp[ly][lx] = pv[q];
            if constexpr (COMP) S.sl[ly][lx] = lv[q];
            if (load_k) S.sk[ly][lx] = kv[q];
            // the tile's own nodes (ring columns that wrap are another tile's)
            if (inside && lx >= 1 && lx <= SX && ly >= 1 && ly <= SY && x0 + lx - 1 < nx) {
                if (e) {
                    psi_new[n] = pv[q];
                    if constexpr (COMP) psi_new[ps + n] = lv[q];
                }
                if (first) A.k0[n] = TC(kv[q]);
            }
        });
    }
    worker_sync<RT>(w);
    long long mx = 0;
    T sum = T(0), ks = T(0);
    auto child = [&](int i, int j, Node9<T> &nd) {
        const int lx = i - x0 + 1, ly = j - y0 + 1;
        const long long n = (long long)j * pitch + i;
        auto pat = [&](int dx, int dy) { return S.sp[ly + dy][lx + dx]; };
        auto kat = [&](int dx, int dy) {  // mirrored at the walls (above the ring's top row too)
            const int gy = j + dy, my = gy < 0 ? 0 : (gy >= ny ? ny - 1 : gy);
            return S.sk[my - y0 + 1][lx + dx];
        };
        T r;
        if constexpr (COMP) {
            auto lat = [&](int dx, int dy) { return S.sl[ly + dy][lx + dx]; };
            nd = node9_pairs<true>(kat, j, ny, A.H0c, A.H0s);
            if (L0.rhs) nd.b = L0.rhs[n];
            r = resid_pairs<true>(nd, pat, lat, j, ny);
        } else {
            if (form) {  // the regrouped sums hold on the walls too, but for psi'(ghost) = -psi'(node)
                nd = node9<T, false>(kat, j, ny, A.H0c, A.H0s);
                if (j == 0) nd.diag += nd.c[4];
                if (j == ny - 1) nd.diag += nd.c[2];
#pragma unroll
                for (int a = 1; a < 9; a++) L0.coef[(a - 1) * ps + n] = nd.c[a];
                L0.coef[8 * ps + n] = nd.diag;
                L0.coef[9 * ps + n] = nd.b;
                if (L0.rhs) nd.b = L0.rhs[n];
            }
            r = nd.b - (off9_two<T>(nd, pat, j, ny) - nd.diag * S.sp[ly][lx]);
        }
        A.r0[n] = unit.of(r);
        sum += r;
        if (first) ks += S.sk[ly][lx];
        mx = max(mx, max_bits(r));
    };
    if (live) {
        child(ia, j0, pre[0]);
        child(ia + 1, j0, pre[PLANES ? 1 : 0]);
    }
    if (third) {
        for (int c = 0; c < 2; c++) {
            Node9<T> nd;
            if (PLANES && !form) coef(nd, ia + c, j0 + 1);
            child(ia + c, j0 + 1, nd);
        }
    }
    if (merged) {  // the cell's other row
        sum += __shfl_xor_sync(0xffffffffu, sum, SX / 2);
        if (first) ks += __shfl_xor_sync(0xffffffffu, ks, SX / 2);
    }
    if (live && (!merged || (tid & (SX / 2)) == 0)) {
        const int I = ia / 2, J = merged ? j0 / 2 : j0;
        const long long q = (long long)J * L1.pitch + I;
        L1.b[q] = unit.of(sum);
        if (first) L1.k[q] = TC(ks / (T(L1.wx[I]) * T(L1.wy[J])));  // unit lattice cells
    }
    worker_sync<RT>(w);
    return mx;
}

// Restriction of level F (pre-smoothed iterate in F.r) onto C, one cell per
// thread: the residuals of its children, all their loads issued first.
__device__ __forceinline__ void restrict_phase(const Level<TC> &F, const Level<TC> &C, bool keep_k) {
    const int nx = F.nx, ny = F.ny, p = F.pitch;
    for (int t = blockIdx.x * SOLVE_THREADS + threadIdx.x; t < C.nx * C.ny; t += gridDim.x * SOLVE_THREADS) {
        const int I = t % C.nx, J = t / C.nx, ia = C.cx0[I], ib = C.cx0[I + 1], ja = C.cy0[J], jb = C.cy0[J + 1];
        TC sr = 0, sk = 0;
        // the w x h block of children from (i0, j0), w, h <= 2, with its neighbours
        auto part = [&](int i0, int j0, int w, int h) {
            TC e[4][4], k[4][4], b[2][2];
#pragma unroll
            for (int y = 0; y < 4; y++)
#pragma unroll
                for (int x = 0; x < 4; x++) {
                    e[y][x] = k[y][x] = 0;
                    const int gy = j0 - 1 + y;
                    int gx = i0 - 1 + x;
                    const bool corner = (x == 0 || x > w) && (y == 0 || y > h);
                    if (corner || x > w + 1 || y > h + 1 || gy < 0 || gy >= ny) continue;
                    gx = gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx);
                    const long long n = (long long)gy * p + gx;
                    e[y][x] = __ldcg(F.r + n);
                    k[y][x] = __ldcg(F.k + n);
                    if (x >= 1 && x <= w && y >= 1 && y <= h) b[y - 1][x - 1] = __ldcg(F.b + n);
                }
#pragma unroll
            for (int y = 0; y < 2; y++)
#pragma unroll
                for (int x = 0; x < 2; x++) {
                    if (x >= w || y >= h) continue;
                    auto kat = [&](int dx, int dy) { return k[y + 1 + dy][x + 1 + dx]; };
                    const FV<TC> f = fv_coef(F, i0 + x, j0 + y, kat);
                    TC s = f.te * e[y + 1][x + 2] + f.tw * e[y + 1][x];
                    if (f.hasn) s += f.tn * e[y + 2][x + 1];
                    if (f.hass) s += f.ts * e[y][x + 1];
                    sr += b[y][x] - (s - (f.te + f.tw + f.tn + f.ts) * e[y + 1][x + 1]);
                    if (keep_k) sk += k[y + 1][x + 1] * F.wx[i0 + x] * F.wy[j0 + y];
                }
        };
        if (ib - ia == 2 && jb - ja == 2) {
            part(ia, ja, 2, 2);
        } else {
            for (int j = ja; j < jb; j++)
                for (int i = ia; i < ib; i++) part(i, j, 1, 1);
        }
        C.b[(long long)J * C.pitch + I] = sr;
        if (keep_k) C.k[(long long)J * C.pitch + I] = sk / (C.wx[I] * C.wy[J]);
    }
}

// Interpolation of level C's correction (another block's values) onto a tile.
template <int NXT, int NYT>
__device__ __forceinline__ TC prolong_cg(const ProlongTile<TC, NXT, NYT> &pt, const Level<TC> &C, int lx, int ly) {
    const int x0 = pt.x0[lx], x1 = pt.x1[lx], y0 = pt.y0[ly], y1 = pt.y1[ly];
    const TC wx = pt.wx[lx], wy = pt.wy[ly];
    TC a = 0, b = 0;
    if (y0 >= 0)
        a = (TC(1) - wx) * __ldcg(C.e + (long long)y0 * C.pitch + x0) + wx * __ldcg(C.e + (long long)y0 * C.pitch + x1);
    if (y1 >= 0)
        b = (TC(1) - wx) * __ldcg(C.e + (long long)y1 * C.pitch + x0) + wx * __ldcg(C.e + (long long)y1 * C.pitch + x1);
    return (TC(1) - wy) * a + wy * b;
}

struct FvTile {
    TC se[FVH + 2][SX + 2], sk[FVH + 2][SX + 2];
    ProlongTile<TC, SX + 2, FVH + 2> pt;
};

// Red-black sweeps of a coarse level, 32 x FVH cells per block with a frozen
// ring (KIND as in fv_smooth_tile).
template <int KIND>
__device__ __forceinline__ void fv_phase(FvTile &S, const Level<TC> &L, const Level<TC> &C, int sweeps) {
    const int nx = L.nx, ny = L.ny, p = L.pitch, tx = threadIdx.x % SX, ty = threadIdx.x / SX;
    const int gx_ = (nx + SX - 1) / SX, gy_ = (ny + FVH - 1) / FVH, ncol = (nx & 1) ? 4 : 2;
    for (int tile = blockIdx.x; tile < gx_ * gy_; tile += gridDim.x) {
        const int x0 = (tile % gx_) * SX, y0 = (tile / gx_) * FVH;
        if (KIND == 1) {
            static_assert(SX + 2 + FVH + 2 <= SOLVE_THREADS, "one thread per table entry");
            const int t = threadIdx.x, q = t - (SX + 2), gy = y0 - 1 + q;
            if (t < SX + 2) {
                int gx = x0 - 1 + t;
                if (gx < 0) gx += nx;
                while (gx >= nx) gx -= nx;
                S.pt.x0[t] = L.px0[gx];
                S.pt.x1[t] = L.px1[gx];
                S.pt.wx[t] = L.pwx[gx];
            } else if (q < FVH + 2) {
                const bool in = gy >= 0 && gy < ny;
                S.pt.y0[q] = in ? L.py0[gy] : -1;
                S.pt.y1[q] = in ? L.py1[gy] : -1;
                S.pt.wy[q] = in ? L.pwy[gy] : TC(0);
            }
            __syncthreads();
        }
#pragma unroll
        for (int q = 0; q < ((SX + 2) * (FVH + 2) + SOLVE_THREADS - 1) / SOLVE_THREADS; q++) {
            const int t = threadIdx.x + q * SOLVE_THREADS;
            if (t >= (SX + 2) * (FVH + 2)) break;
            const int lx = t % (SX + 2), ly = t / (SX + 2), gy = y0 - 1 + ly;
            int gx = x0 - 1 + lx;
            if (gx < 0) gx += nx;
            while (gx >= nx) gx -= nx;
            TC kv = 0, ev = 0;
            if (gy >= 0 && gy < ny) {
                kv = __ldcg(L.k + (long long)gy * p + gx);
                if (KIND == 1) ev = __ldcg(L.r + (long long)gy * p + gx) + prolong_cg(S.pt, C, lx, ly);
            }
            S.sk[ly][lx] = kv;
            S.se[ly][lx] = ev;
        }
        __syncthreads();
        const int lx = tx + 1, ly = ty + 1, I = x0 + tx, J = y0 + ty;
        const bool own = I < nx && J < ny;
        FV<TC> f;
        TC idg = 0, b = 0;
        if (own) {
            auto kat = [&](int dx, int dy) { return S.sk[ly + dy][lx + dx]; };
            f = fv_coef(L, I, J, kat);
            idg = TC(1) / (f.te + f.tw + f.tn + f.ts);
            b = __ldcg(L.b + (long long)J * p + I);
        }
        const int colour = own ? fv_colour(I, J, nx) : -1;
        for (int s = 0; s < sweeps; s++)
            for (int c = 0; c < ncol; c++) {
                if (colour == c) {
                    TC v = f.te * S.se[ly][lx + 1] + f.tw * S.se[ly][lx - 1];
                    if (f.hasn) v += f.tn * S.se[ly + 1][lx];
                    if (f.hass) v += f.ts * S.se[ly - 1][lx];
                    S.se[ly][lx] = (v - b) * idg;
                }
                __syncthreads();
            }
        if (own) (KIND == 0 ? L.r : L.e)[(long long)J * p + I] = S.se[ly][lx];
        __syncthreads();
    }
}

// Division by a level's width or half width: x / d = (x * ceil(2^32 / d)) >> 32
// for x, d < 2^16 (the single-block levels hold at most SOLVE_CELLS cells).
static_assert(SOLVE_CELLS < 65536, "magic division of cell indices");
__device__ __forceinline__ int quot(int x, unsigned m) { return (int)__umulhi((unsigned)x, m); }
__device__ __forceinline__ unsigned quot_magic(int d) {
    return d <= 1 ? 0u : (unsigned)((0x100000000ull + (unsigned)d - 1) / (unsigned)d);
}

// One of the single-block levels in block 0's shared memory: correction,
// right-hand side, east and north face coefficients, reciprocal diagonal.
constexpr int BOTTOM_ARRAYS = 5;
struct Bottom {
    int nx, ny, pairs;  // pairs of columns (the odd last one has its own colours)
    unsigned mnx, mpairs;
    int at;             // first of its arrays, in values from the block's bottom storage
};
// its arrays as pointers into shared memory (a copy: nothing is reloaded)
struct BottomView {
    int nx, ny, pairs;
    unsigned mnx, mpairs;
    TC *__restrict__ e, *__restrict__ b, *__restrict__ te, *__restrict__ tn, *__restrict__ dg;
    __device__ __forceinline__ BottomView(TC *sm, const Bottom &B)
        : nx(B.nx), ny(B.ny), pairs(B.pairs), mnx(B.mnx), mpairs(B.mpairs) {
        const int n = nx * ny;
        e = sm + B.at;
        b = e + n;
        te = b + n;
        tn = te + n;
        dg = tn + n;
    }
};

// One colour of a red-black sweep (colours 2 and 3: the odd last column's rows).
// ZERO: the iterate is still 0 in every neighbour (first colour of a pre-sweep).
template <bool ZERO>
__device__ __forceinline__ void bottom_colour(const BottomView &B, int c, int t0, int nthr) {
    const int nx = B.nx, ny = B.ny;
    const int n = c < 2 ? B.pairs * ny : (ny + 3 - c) / 2;
#pragma unroll 2
    for (int u = t0; u < n; u += nthr) {
        int I, J;
        if (c < 2) {
            J = B.pairs > 1 ? quot(u, B.mpairs) : u;
            I = 2 * (u - J * B.pairs) + ((J + c) & 1);
        } else {
            I = nx - 1;
            J = 2 * u + c - 2;
        }
        const int t = J * nx + I;
        TC v = 0;
        if (!ZERO) {
            const int tw = I == 0 ? t + nx - 1 : t - 1, te = I + 1 == nx ? t + 1 - nx : t + 1;
            v = B.te[t] * B.e[te] + B.te[tw] * B.e[tw];
            if (J + 1 < ny) v += B.tn[t] * B.e[t + nx];
            if (J > 0) v += B.tn[t - nx] * B.e[t - nx];
        }
        B.e[t] = (v - B.b[t]) * B.dg[t];
    }
}

// sync: __syncthreads, or __syncwarp where one warp does the level.
template <typename F>
__device__ __forceinline__ void bottom_sweeps(const BottomView &B, int sweeps, bool from_zero, int t0, int nthr, F sync) {
    const int ncol = (B.nx & 1) ? 4 : 2;
    for (int s = 0; s < sweeps; s++)
        for (int c = 0; c < ncol; c++) {
            if (from_zero && s == 0 && c == 0) bottom_colour<true>(B, c, t0, nthr);
            else bottom_colour<false>(B, c, t0, nthr);
            sync();
        }
}

// NU_COARSEST sweeps of the last level (at most MIN_COARSE cells) from zero by
// one warp: a lane keeps the coefficients of its two cells of either colour (and
// its one of the odd last column) in registers, so that a colour is one round of
// shared-memory loads. The colours are those of bottom_colour.
static_assert(MIN_COARSE <= 128, "two cells of a colour per lane");
__device__ __forceinline__ void bottom_last(const BottomView &B) {
    const int nx = B.nx, ny = B.ny, lane = threadIdx.x;
    constexpr int CELLS = 6;  // colour 0: 0, 1; colour 1: 2, 3; colours 2, 3: 4, 5
    TC ce[CELLS], cw[CELLS], cn[CELLS], cs[CELLS], dg[CELLS], bd[CELLS];
    int at[CELLS], te[CELLS], tw[CELLS], tn[CELLS], ts[CELLS];
    bool has[CELLS];
    const int half = B.pairs * ny;
#pragma unroll
    for (int i = 0; i < CELLS; i++) {
        const int c = i < 4 ? i >> 1 : i - 2, u = i < 4 ? lane + 32 * (i & 1) : lane;
        int I, J;
        if (i < 4) {
            has[i] = u < half;
            J = has[i] ? (B.pairs > 1 ? quot(u, B.mpairs) : u) : 0;
            I = has[i] ? 2 * (u - J * B.pairs) + ((J + c) & 1) : 0;
        } else {
            has[i] = (nx & 1) && 2 * u + c - 2 < ny;
            J = has[i] ? 2 * u + c - 2 : 0;
            I = nx - 1;
        }
        const int t = J * nx + I;
        at[i] = t;
        te[i] = I + 1 == nx ? t + 1 - nx : t + 1;
        tw[i] = I == 0 ? t + nx - 1 : t - 1;
        tn[i] = J + 1 < ny ? t + nx : t;
        ts[i] = J > 0 ? t - nx : t;
        dg[i] = B.dg[t];
        ce[i] = B.te[t] * dg[i];
        cw[i] = B.te[tw[i]] * dg[i];
        cn[i] = J + 1 < ny ? B.tn[t] * dg[i] : TC(0);
        cs[i] = J > 0 ? B.tn[t - nx] * dg[i] : TC(0);
        bd[i] = B.b[t] * dg[i];
    }
    auto update = [&](int i) {
        return (ce[i] * B.e[te[i]] + cw[i] * B.e[tw[i]]) + (cn[i] * B.e[tn[i]] + cs[i] * B.e[ts[i]]) - bd[i];
    };
    for (int s = 0; s < NU_COARSEST; s++) {
#pragma unroll
        for (int c = 0; c < 2; c++) {
            const TC v0 = update(2 * c), v1 = update(2 * c + 1);
            if (has[2 * c]) B.e[at[2 * c]] = v0;
            if (has[2 * c + 1]) B.e[at[2 * c + 1]] = v1;
            __syncwarp();
        }
        if (nx & 1) {
#pragma unroll
            for (int i = 4; i < 6; i++) {
                const TC v = update(i);
                if (has[i]) B.e[at[i]] = v;
                __syncwarp();
            }
        }
    }
}

// Levels lc .. nl - 1 of a V-cycle (V(1,1), NU_COARSEST sweeps on the last)
// inside block 0, whose shared memory keeps them for the whole solve; setup: the
// first cycle, which also forms their permeabilities and coefficients.
__device__ __forceinline__ void bottom_phase(TC *sm, const Bottom *B, const Level<TC> *L, int lc, int nl, bool setup) {
    const int tid = threadIdx.x;
    constexpr int nthr = SOLVE_THREADS;
    auto all = [] { __syncthreads(); };
    if (setup) {  // the permeabilities go through e
        const BottomView V(sm, B[lc]);
        for (int t = tid; t < V.nx * V.ny; t += nthr) V.e[t] = __ldcg(L[lc].k + t);  // pitch = nx
        __syncthreads();
        for (int l = lc + 1; l < nl; l++) {
            const BottomView F(sm, B[l - 1]), V2(sm, B[l]);
            const Level<TC> &C = L[l], &Fl = L[l - 1];
            for (int t = tid; t < V2.nx * V2.ny; t += nthr) {
                const int J = quot(t, V2.mnx), I = t - J * V2.nx;
                TC s = 0;
                for (int j = C.cy0[J]; j < C.cy0[J + 1]; j++)
                    for (int i = C.cx0[I]; i < C.cx0[I + 1]; i++) s += F.e[j * F.nx + i] * Fl.wx[i] * Fl.wy[j];
                V2.e[t] = s / (C.wx[I] * C.wy[J]);
            }
            __syncthreads();
        }
        for (int l = lc; l < nl; l++) {
            const BottomView V2(sm, B[l]);
            const int nx = V2.nx;
            for (int t = tid; t < nx * V2.ny; t += nthr) {
                const int J = quot(t, V2.mnx), I = t - J * nx;
                auto kat = [&](int dx, int dy) {
                    int ii = I + dx;
                    ii = ii < 0 ? nx - 1 : (ii >= nx ? 0 : ii);
                    return V2.e[(J + dy) * nx + ii];
                };
                const FV<TC> f = fv_coef(L[l], I, J, kat);
                V2.te[t] = f.te;
                V2.tn[t] = f.tn;
                V2.dg[t] = TC(1) / (f.te + f.tw + f.tn + f.ts);
            }
        }
        __syncthreads();
    }
    {
        const BottomView V(sm, B[lc]);
        constexpr int Q = ((int)SOLVE_CELLS + nthr - 1) / nthr;
        TC v[Q];
        const TC *const src = L[lc].b;
#pragma unroll
        for (int q = 0; q < Q; q++) v[q] = tid + q * nthr < V.nx * V.ny ? __ldcg(src + tid + q * nthr) : TC(0);
#pragma unroll
        for (int q = 0; q < Q; q++)
            if (tid + q * nthr < V.nx * V.ny) {
                V.b[tid + q * nthr] = v[q];
                V.e[tid + q * nthr] = 0;
            }
        __syncthreads();
    }
    for (int l = lc; l < nl - 1; l++) {
        const BottomView F(sm, B[l]), V(sm, B[l + 1]);
        bottom_sweeps(F, NU_CTA, true, tid, nthr, all);
        const int nx = F.nx, ny = F.ny;
        for (int t = tid; t < V.nx * V.ny; t += nthr) {
            const int J = quot(t, V.mnx), I = t - J * V.nx;
            // children: pairs, the last of an odd count three (merge_faces)
            const int ia = V.nx == nx ? I : 2 * I, ja = V.ny == ny ? J : 2 * J;
            const int ib = I == V.nx - 1 ? nx : (V.nx == nx ? ia + 1 : ia + 2);
            const int jb = J == V.ny - 1 ? ny : (V.ny == ny ? ja + 1 : ja + 2);
            TC s = 0;
            auto child = [&](int i, int j) {
                const int q = j * nx + i;
                const int qw = i == 0 ? q + nx - 1 : q - 1, qe = i + 1 == nx ? q + 1 - nx : q + 1;
                TC v = F.te[q] * F.e[qe] + F.te[qw] * F.e[qw];
                if (j + 1 < ny) v += F.tn[q] * F.e[q + nx];
                if (j > 0) v += F.tn[q - nx] * F.e[q - nx];
                s += F.b[q] - (v - __fdividef(F.e[q], F.dg[q]));
            };
            if (ib - ia == 2 && jb - ja == 2) {
#pragma unroll
                for (int c = 0; c < 4; c++) child(ia + (c & 1), ja + (c >> 1));
            } else {
                for (int j = ja; j < jb; j++)
                    for (int i = ia; i < ib; i++) child(i, j);
            }
            V.b[t] = s;
            V.e[t] = 0;
        }
        __syncthreads();
    }
    if (tid < 32) bottom_last(BottomView(sm, B[nl - 1]));
    __syncthreads();
    for (int l = nl - 2; l >= lc; l--) {
        const BottomView F(sm, B[l]), V(sm, B[l + 1]);
        const int *const px0 = L[l].px0, *const px1 = L[l].px1, *const py0 = L[l].py0, *const py1 = L[l].py1;
        const TC *const pwx = L[l].pwx, *const pwy = L[l].pwy;
#pragma unroll 2
        for (int t = tid; t < F.nx * F.ny; t += nthr) {
            const int j = quot(t, F.mnx), i = t - j * F.nx;
            const int xa = px0[i], xb = px1[i], ya = py0[j], yb = py1[j];
            const TC wx = pwx[i], wy = pwy[j];
            TC a = 0, b = 0;
            if (ya >= 0) a = (TC(1) - wx) * V.e[ya * V.nx + xa] + wx * V.e[ya * V.nx + xb];
            if (yb >= 0) b = (TC(1) - wx) * V.e[yb * V.nx + xa] + wx * V.e[yb * V.nx + xb];
            F.e[t] += (TC(1) - wy) * a + wy * b;
        }
        __syncthreads();
        bottom_sweeps(F, NU_CTA, false, tid, nthr, all);
    }
    const BottomView V(sm, B[lc]);
    TC *const dst = L[lc].e;
    for (int t = tid; t < V.nx * V.ny; t += nthr) dst[t] = V.e[t];
}

template <typename T, bool COMP>
union SolveTile {
    ResidTile<T, COMP> r;
    SweepTile s;
};

template <typename T, bool COMP>
__host__ __device__ constexpr size_t solve_tiles_bytes() {
    const size_t a = SOLVE_WORKERS * sizeof(SolveTile<T, COMP>), b = sizeof(FvTile);
    return ((a > b ? a : b) + 15) / 16 * 16;
}

template <typename T, bool COMP>
__global__ void __launch_bounds__(SOLVE_THREADS, 1) mg_solve_kernel(const SolveArgs<T> A) {
    extern __shared__ __align__(16) unsigned char raw[];
    SolveTile<T, COMP> *wt = reinterpret_cast<SolveTile<T, COMP> *>(raw);
    FvTile &fv = *reinterpret_cast<FvTile *>(raw);
    TC *bottom = reinterpret_cast<TC *>(raw + solve_tiles_bytes<T, COMP>());
    __shared__ Level<TC> L[MAX_LEVELS];
    __shared__ Bottom B[MAX_LEVELS];
    __shared__ long long wmax[SOLVE_THREADS / 32];
    __shared__ double norm;
    MgCtl *const ctl = A.ctl;
    const int tid = threadIdx.x, nl = A.nl, lc = A.lc;
    __shared__ int given_up;  // one answer for the block: a solve beside this one may give up right now
    const unsigned polls = A.bound->polls;
    if (tid < nl) L[tid] = A.lv[tid];
    if (tid == 0) given_up = *(volatile int *)&A.bound->stuck;
    __syncthreads();
    if (given_up) return;  // a barrier of this context timed out
    if (tid == 0) {
        int at = 0;
        for (int l = lc; l < nl; l++) {
            B[l] = Bottom{L[l].nx, L[l].ny, L[l].nx / 2, quot_magic(L[l].nx), quot_magic(L[l].nx / 2), at};
            at += BOTTOM_ARRAYS * L[l].nx * L[l].ny;
        }
    }
    __syncthreads();
    const int gx = (A.L0.nx + SX - 1) / SX, tiles = gx * ((A.L0.ny + SY - 1) / SY);
    const double tol = ctl->tolH0, stop = COMP ? tol : ctl->stop;
    const Unit<T> unit(ctl->scale);
    const int max_iter = ctl->max_iter;
    int cur = ctl->cur, iter = 0, heads = 0, twogrid = 0, vcycles = 0;
    unsigned arrivals = 0;
    bool closing = false;          // the tolerance is met
    double res = 0.0, last = 0.0;  // max |r| of psi(cur); of the closing head before
    const TC over = L[1].ny != A.L0.ny && A.L0.ny % 2 == 0 ? OVER : TC(1);
    auto psi = [&](int c) { return c ? A.L0.r : A.L0.e; };
    // tile t is worker (t / gridDim) % workers of block t % gridDim
    auto each_tile = [&](int w, int workers, auto f) {
        for (int t = blockIdx.x + w * gridDim.x; t < tiles; t += workers * gridDim.x) f(t % gx, t / gx);
    };
    const int rw = tid / RT, rt = tid % RT, sw = tid / QT, st = tid % QT;
    while (true) {
        long long mx = 0;
        each_tile(rw, RESID_WORKERS, [&](int bx, int by) {
            mx = max(mx, resid_tile<T, COMP>(wt[rw].r, A, L[1], psi(cur), psi(cur ^ 1), iter ? A.eB : nullptr, unit,
                                             heads == 0, bx, by, rw, rt));
        });
        if (iter) cur ^= 1;
        for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if ((tid & 31) == 0) wmax[tid >> 5] = mx;
        __syncthreads();
        if (tid == 0) {
#pragma unroll
            for (int q = 1; q < SOLVE_THREADS / 32; q++) mx = max(mx, wmax[q]);
            if (mx > 0) atomic_max_nonneg(&ctl->norm_slot[heads & 3], max_value(mx, T(0)));
        }
        if (!grid_barrier(ctl, A.bound, polls, arrivals)) return;
        if (tid == 0) {
            norm = __longlong_as_double((long long)__ldcg(&ctl->norm_slot[heads & 3]));
            if (blockIdx.x == 0) ctl->norm_slot[(heads + 2) & 3] = 0ull;  // two heads on, two barriers away
        }
        __syncthreads();
        heads++;
        res = norm;
        if (closing && !(res < last)) {  // only rounding was left: the iterate before is the better one
            cur ^= 1;
            res = last;
            break;
        }
        if (res <= stop || iter >= max_iter || !(res < INFINITY)) break;
        if (res <= tol) {
            if (closing && res > 0.5 * last) break;
            closing = true;
            last = res;
        }
        if (twogrid < 2) {
            twogrid++;
            fv_phase<2>(fv, L[1], L[1], NU_TWOGRID);
        } else {
            const bool setup = vcycles++ == 0;
            for (int l = 1; l < lc; l++) {
                fv_phase<0>(fv, L[l], L[l + 1], NU_PRE);
                if (!grid_barrier(ctl, A.bound, polls, arrivals)) return;
                restrict_phase(L[l], L[l + 1], setup);
                if (!grid_barrier(ctl, A.bound, polls, arrivals)) return;
            }
            if (blockIdx.x == 0) bottom_phase(bottom, B, L, lc, nl, setup);
            for (int l = lc - 1; l >= 1; l--) {
                if (!grid_barrier(ctl, A.bound, polls, arrivals)) return;
                fv_phase<1>(fv, L[l], L[l + 1], NU_POST);
            }
        }
        if (!grid_barrier(ctl, A.bound, polls, arrivals)) return;
        each_tile(sw, SOLVE_WORKERS, [&](int bx, int by) { sweep_tile<T>(wt[sw].s, A, L[1], nullptr, A.eA, TC(1), bx, by, sw, st); });
        if (!grid_barrier(ctl, A.bound, polls, arrivals)) return;
        each_tile(sw, SOLVE_WORKERS, [&](int bx, int by) { sweep_tile<T>(wt[sw].s, A, L[1], A.eA, A.eB, over, bx, by, sw, st); });
        if (!grid_barrier(ctl, A.bound, polls, arrivals)) return;
        iter++;
    }
    if (blockIdx.x == 0 && tid == 0) {
        ctl->done = 1;
        ctl->keep_going = 0;
        ctl->mode = 3;
        ctl->iter = iter;
        ctl->cur = cur;
        ctl->converged = res <= tol;
        if (!(res <= tol)) ctl->nonconv_count++;
        ctl->last_resid = ctl->H0 > 0.0 ? res / ctl->H0 : 0.0;
        ctl->last_iters = iter;
        ctl->cycles_launched += heads;
        ctl->total_cycles += vcycles;
        ctl->twogrid_cycles += twogrid;
    }
}

}  // namespace fcd
