// Kernels of the continuous Q1 levels of the hp hierarchy (paper Sec. 2.4 and
// Sec. 5.2): the vertex gather of the p-restriction, damped point Jacobi with
// the 3^d-point Galerkin stencils, residual, nested h-restriction and
// h-prolongation, and the dense coarsest solve.
#include <algorithm>

#include "internal.h"

namespace dgmg {

namespace {

constexpr int TPB = 256;

template <int DIM>
__device__ __forceinline__ void vcoords(int64_t v, const int *m, int *c) {
    if (v <= 0x7fffffff) {   // 32-bit division where it suffices
        const unsigned u = (unsigned)v, m0 = (unsigned)m[0], r = u / m0;
        c[0] = (int)(u - r * m0);
        if (DIM == 3) {
            const unsigned m1 = (unsigned)m[1], z = r / m1;
            c[1] = (int)(r - z * m1);
            c[2] = (int)z;
        } else {
            c[1] = (int)r;
        }
        return;
    }
    c[0] = (int)(v % m[0]);
    const int64_t r = v / m[0];
    if (DIM == 3) {
        c[1] = (int)(r % m[1]);
        c[2] = (int)(r / m[1]);
    } else {
        c[1] = (int)r;
    }
}

// b0[v] = sum over the 2^d cells around interior vertex v of the cell's corner
// partial sum for that vertex (fixed order: deterministic p-restriction).
template <int DIM, typename T>
__device__ __forceinline__ T corner_sum_at(int n0, int n1, int n2, const T *__restrict__ corners, int64_t v) {
    const int m[3] = {n0 - 1, n1 - 1, n2 - 1};
    int c[3];
    vcoords<DIM>(v, m, c);
    T s = T(0);
#pragma unroll
    for (int a = 0; a < (1 << DIM); ++a) {
        // cell with lower corner (vertex - 1 + a) along each axis; the vertex is
        // that cell's corner (1 - a) along each axis
        const int cx = c[0] + (a & 1), cy = c[1] + ((a >> 1) & 1), cz = DIM == 3 ? c[2] + ((a >> 2) & 1) : 0;
        const int64_t cell = cx + (int64_t)n0 * (cy + (int64_t)n1 * cz);
        const int corner = (~a) & ((1 << DIM) - 1);
        s += corners[cell * (1 << DIM) + corner];
    }
    return s;
}

template <int DIM, typename T>
__device__ __forceinline__ void corner_gather_at(int n0, int n1, int n2, const T *__restrict__ corners,
                                                 T *__restrict__ b0, int64_t v) {
    const int64_t nv = DIM == 3 ? (int64_t)(n0 - 1) * (n1 - 1) * (n2 - 1) : (int64_t)(n0 - 1) * (n1 - 1);
    if (v < nv) b0[v] = corner_sum_at<DIM, T>(n0, n1, n2, corners, v);
}

template <int DIM, typename T>
__global__ void k_corner_gather(int n0, int n1, int n2, const T *__restrict__ corners, T *__restrict__ b0) {
    corner_gather_at<DIM, T>(n0, n1, n2, corners, b0, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// (A u)[v] with the 3^d-point stencil. All loads are issued before the
// products, so that a vertex costs one memory round trip, not one per point.
template <int DIM, typename T>
__device__ __forceinline__ T stencil_apply(const CGLevelDev<T> &L, int64_t v, const int *c, const T *u) {
    constexpr int NS = DIM == 3 ? 27 : 9;
    T sv[NS], uv[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        const int sx = k % 3 - 1, sy = (k / 3) % 3 - 1, sz = DIM == 3 ? k / 9 - 1 : 0;
        const int x = c[0] + sx, y = c[1] + sy, z = DIM == 3 ? c[2] + sz : 0;
        const bool in = x >= 0 && x < L.m[0] && y >= 0 && y < L.m[1] && (DIM == 2 || (z >= 0 && z < L.m[2]));
        const int64_t w = x + (int64_t)L.m[0] * (y + (int64_t)L.m[1] * z);
        sv[k] = in ? __ldg(L.st + (int64_t)k * L.nv + v) : T(0);
        uv[k] = in ? u[w] : T(0);
    }
    T s[3] = {};   // three chains of dependent sums
#pragma unroll
    for (int k = 0; k < NS; ++k) s[k / (NS / 3)] += sv[k] * uv[k];
    return (s[0] + s[1]) + s[2];
}

template <int DIM, typename T>
__device__ __forceinline__ void cg_jacobi_at(const CGLevelDev<T> &L, const T *u_in,
                                             const T *b, T *u_out, T omega,
                                             int zero_guess, int64_t v) {
    constexpr int NS = DIM == 3 ? 27 : 9;
    if (v >= L.nv) return;
    const T diag = __ldg(L.st + (int64_t)(NS / 2) * L.nv + v);
    if (zero_guess) {
        u_out[v] = omega * b[v] / diag;
        return;
    }
    int c[3] = {0, 0, 0};
    vcoords<DIM>(v, L.m, c);
    const T au = stencil_apply<DIM, T>(L, v, c, u_in);
    u_out[v] = u_in[v] + omega * (b[v] - au) / diag;
}

template <int DIM, typename T>
__global__ void k_cg_jacobi(CGLevelDev<T> L, const T *__restrict__ u_in, const T *__restrict__ b,
                            T *__restrict__ u_out, T omega, int zero_guess) {
    cg_jacobi_at<DIM, T>(L, u_in, b, u_out, omega, zero_guess, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

template <int DIM, typename T>
__device__ __forceinline__ void cg_residual_at(const CGLevelDev<T> &L, const T *u,
                                               const T *b, T *r, int64_t v) {
    if (v >= L.nv) return;
    int c[3] = {0, 0, 0};
    vcoords<DIM>(v, L.m, c);
    r[v] = b[v] - stencil_apply<DIM, T>(L, v, c, u);
}

template <int DIM, typename T>
__global__ void k_cg_residual(CGLevelDev<T> L, const T *__restrict__ u, const T *__restrict__ b,
                              T *__restrict__ r) {
    cg_residual_at<DIM, T>(L, u, b, r, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// sum_i P_h[i][V] rf[i]: per axis, the fine children of coarse vertex V, at most
// 2f - 1 <= 5 (weights padded to 5). Eight lanes share a vertex, each takes every
// eighth of its rows of children along x: the rows' loads are all in flight and the
// chain of dependent sums is short (one thread per vertex took 5.4 us a level in FP64,
// against 3.2 of a Jacobi step). All 32 lanes of a warp call it; V < 0: no vertex.
// Every lane of a group returns the sum.
constexpr int RS_LANES = 8;
template <int DIM, typename T>
__device__ __forceinline__ T h_restrict_at(const CGLevelDev<T> &L, const T *rf, int64_t V) {
    constexpr int ROWS = DIM == 3 ? 25 : 5, R = (ROWS + RS_LANES - 1) / RS_LANES;
    const int lane = threadIdx.x & (RS_LANES - 1);
    T s = T(0);
    if (V >= 0) {
        int C[3] = {0, 0, 0};
        vcoords<DIM>(V, L.mc, C);
        const int sx = __ldg(L.rs_start[0] + C[0]), nx = __ldg(L.rs_cnt[0] + C[0]);
        const int sy = __ldg(L.rs_start[1] + C[1]), ny = __ldg(L.rs_cnt[1] + C[1]);
        const int sz = DIM == 3 ? __ldg(L.rs_start[2] + C[2]) : 0, nz = DIM == 3 ? __ldg(L.rs_cnt[2] + C[2]) : 1;
        T wx[5], w[R], f[R][5];
#pragma unroll
        for (int i = 0; i < 5; ++i) wx[i] = __ldg(L.rs_w[0] + C[0] * 5 + i);
#pragma unroll
        for (int a = 0; a < R; ++a) {
            const int row = lane + a * RS_LANES, k = DIM == 3 ? row / 5 : 0, j = DIM == 3 ? row - 5 * k : row;
            const bool in = row < ROWS && j < ny && k < nz;
            w[a] = in ? __ldg(L.rs_w[1] + C[1] * 5 + j) : T(0);
            if (DIM == 3 && in) w[a] *= __ldg(L.rs_w[2] + C[2] * 5 + k);
            const T *x = rf + (int64_t)L.m[0] * ((sy + j) + (int64_t)L.m[1] * (sz + k)) + sx;
#pragma unroll
            for (int i = 0; i < 5; ++i) f[a][i] = in && i < nx ? x[i] : T(0);
        }
#pragma unroll
        for (int a = 0; a < R; ++a) {
            T sr = T(0);
#pragma unroll
            for (int i = 0; i < 5; ++i) sr += wx[i] * f[a][i];
            s += w[a] * sr;
        }
    }
#pragma unroll
    for (int o = RS_LANES / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

template <int DIM, typename T>
__global__ void k_h_restrict(CGLevelDev<T> L, const T *__restrict__ rf, T *__restrict__ rc) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, V = t / RS_LANES;
    const bool in = V < (DIM == 3 ? (int64_t)L.mc[0] * L.mc[1] * L.mc[2] : (int64_t)L.mc[0] * L.mc[1]);
    const T s = h_restrict_at<DIM, T>(L, rf, in ? V : -1);
    if (in && t % RS_LANES == 0) rc[V] = s;
}

// uf[i] += sum_V P_h[i][V] ec[V]: per axis, the (at most two) coarse parents.
template <int DIM, typename T>
__device__ __forceinline__ void h_prolong_at(const CGLevelDev<T> &L, const T *ec, T *uf,
                                             int64_t v) {
    if (v >= L.nv) return;
    int c[3] = {0, 0, 0};
    vcoords<DIM>(v, L.m, c);
    int px[2] = {L.pl_lo[0][c[0]], L.pl_hi[0][c[0]]};
    T wx[2] = {L.pl_wlo[0][c[0]], L.pl_whi[0][c[0]]};
    int py[2] = {L.pl_lo[1][c[1]], L.pl_hi[1][c[1]]};
    T wy[2] = {L.pl_wlo[1][c[1]], L.pl_whi[1][c[1]]};
    int pz[2] = {0, -1};
    T wz[2] = {T(1), T(0)};
    if (DIM == 3) {
        pz[0] = L.pl_lo[2][c[2]];
        pz[1] = L.pl_hi[2][c[2]];
        wz[0] = L.pl_wlo[2][c[2]];
        wz[1] = L.pl_whi[2][c[2]];
    }
    T e[8];   // the (up to 8) parents, loaded before they are summed
#pragma unroll
    for (int n = 0; n < 8; ++n) {
        const int i = n & 1, j = (n >> 1) & 1, k = n >> 2;
        e[n] = (px[i] >= 0 && py[j] >= 0 && pz[k] >= 0)
                   ? ec[px[i] + (int64_t)L.mc[0] * (py[j] + (int64_t)L.mc[1] * pz[k])]
                   : T(0);
    }
    T s = T(0);
#pragma unroll
    for (int n = 0; n < 8; ++n) {
        const int i = n & 1, j = (n >> 1) & 1, k = n >> 2;
        if (px[i] >= 0 && py[j] >= 0 && pz[k] >= 0) s += wx[i] * wy[j] * wz[k] * e[n];
    }
    uf[v] += s;
}

template <int DIM, typename T>
__global__ void k_h_prolong(CGLevelDev<T> L, const T *__restrict__ ec, T *__restrict__ uf) {
    h_prolong_at<DIM, T>(L, ec, uf, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// e = A_c^{-1} r with the explicit FP64 inverse of the coarsest operator.
template <typename T>
__device__ __forceinline__ void coarse_row(int64_t nc, const double *Ainv, const T *r,
                                           T *e, int64_t i) {
    if (i >= nc) return;
    // four partial sums: four loads of the row in flight at a time
    const double *a = Ainv + i * nc;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    int64_t j = 0;
    for (; j + 4 <= nc; j += 4) {
        s0 += __ldg(a + j) * (double)r[j];
        s1 += __ldg(a + j + 1) * (double)r[j + 1];
        s2 += __ldg(a + j + 2) * (double)r[j + 2];
        s3 += __ldg(a + j + 3) * (double)r[j + 3];
    }
    for (; j < nc; ++j) s0 += __ldg(a + j) * (double)r[j];
    e[i] = (T)((s0 + s1) + (s2 + s3));
}

template <typename T>
__global__ void k_coarse_solve(int64_t nc, const double *__restrict__ Ainv, const T *__restrict__ r,
                               T *__restrict__ e) {
    coarse_row<T>(nc, Ainv, r, e, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

// ---- the whole Q1 h-cycle of one problem in one launch. The cycle is a chain of
// short steps, so their number and the wait between two of them are what it costs: on
// the levels [0, dense_from) every step is a loop over the level's vertices split among
// the blocks of a cooperative grid, separated by a grid-wide barrier; the cycle on
// level dense_from and everything below it is one product with its matrix, which
// k_q1_dense_matrix computes at set-up column by column with the very steps it
// replaces (it is the inverse of the coarsest operator where that level is the last).
// The gather of the right-hand side is the first step, and whoever writes a level's
// right-hand side writes the first Jacobi step from the zero iterate with it.
// The vectors are written and read again inside the one launch, so the per-vertex
// bodies take them through plain pointers (no __restrict__: no loads through the
// non-coherent read-only cache); only the stencils and tables use __ldg.

// Waits of the grid barrier that gave up (zero in every healthy run). Once one
// has, every later cycle launch returns at once: its output is then not to be
// trusted, and this counter (part of dgmg_wait_timeouts) says so.
__device__ unsigned long long g_q1_barrier_timeouts;

__device__ __forceinline__ unsigned long long ld_acquire_gpu(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long atom_add_acq_rel_gpu(unsigned long long *p, unsigned long long v) {
    unsigned long long old;
    asm volatile("atom.acq_rel.gpu.global.add.u64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v) : "memory");
    return old;
}

// Grid-wide barrier of a co-resident (cooperative) grid on a 64-bit arrival
// counter that only grows: every launch on it has the same number of blocks B
// and passes all its barriers, so the counter is a multiple of B when a launch
// starts and barrier k of the launch is passed once it reaches base + (k+1) B
// (base read off the first arrival). One read-modify-write with release and
// acquire order per block, then polling reads with acquire order: the writes
// of the whole grid before the barrier are visible after it. The wait is
// bounded (about a second); a wait that runs out is counted.
struct GridSync {
    unsigned long long *cnt;
    unsigned long long base;
    unsigned k;
    __device__ __forceinline__ void operator()() {
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned long long o = atom_add_acq_rel_gpu(cnt, 1ull);
            if (k == 0) base = o - o % gridDim.x;
            const unsigned long long target = base + (unsigned long long)(k + 1) * gridDim.x;
            if (o + 1 != target) {
                int it = 0;
                while ((long long)(ld_acquire_gpu(cnt) - target) < 0 && ++it < (1 << 20)) {}
                if (it >= (1 << 20)) atomicAdd(&g_q1_barrier_timeouts, 1ull);
            }
        }
        ++k;
        __syncthreads();
    }
};
struct BlockSync {
    __device__ __forceinline__ void operator()() const { __syncthreads(); }
};

// Work split of one step: on the whole grid every block takes an equal run of
// consecutive warps of items (the runs differ by one warp, so a level of a few
// thousand vertices spreads over all SMs: FP64 FMA throughput per SM is low); in one
// block the threads stride through all.
struct GridEach {
    template <typename F>
    __device__ __forceinline__ void operator()(int64_t n, F &&f) const {
        const int64_t w = (n + 31) / 32, b = w * blockIdx.x / gridDim.x * 32, e = w * (blockIdx.x + 1) / gridDim.x * 32;
        for (int64_t v = b + threadIdx.x; v < (e < n ? e : n); v += blockDim.x) f(v);
    }
    // the same for all lanes of every warp that has an item (f is given v >= n too)
    template <typename F>
    __device__ __forceinline__ void warps(int64_t n, F &&f) const {
        const int64_t w = (n + 31) / 32, b = w * blockIdx.x / gridDim.x * 32, e = w * (blockIdx.x + 1) / gridDim.x * 32;
        for (int64_t v = b + threadIdx.x; v < e; v += blockDim.x) f(v);
    }
};
struct BlockEach {
    template <typename F>
    __device__ __forceinline__ void operator()(int64_t n, F &&f) const {
        for (int64_t v = threadIdx.x; v < n; v += blockDim.x) f(v);
    }
    template <typename F>
    __device__ __forceinline__ void warps(int64_t n, F &&f) const {
        for (int64_t v = threadIdx.x; v < (n + 31) / 32 * 32; v += blockDim.x) f(v);
    }
};

// right-hand side s of vertex v on level l, and the level's first iterate: one Jacobi
// step from zero (u1), or zero (u0) without pre-smoothing
template <typename T>
__device__ __forceinline__ void q1_put_rhs(const Q1Plan<T> &p, int l, int64_t v, T s) {
    p.b[l][v] = s;
    if (p.nu_pre > 0)
        p.u1[l][v] = s * p.wd[l][v];
    else
        p.u0[l][v] = T(0);
}

template <int DIM, typename T>
__device__ __forceinline__ void q1_jacobi_at(const Q1Plan<T> &p, int l, const T *u_in, T *u_out, int64_t v) {
    const CGLevelDev<T> &L = p.L[l];
    int c[3] = {0, 0, 0};
    vcoords<DIM>(v, L.m, c);
    const T w = __ldg(p.wd[l] + v), bv = p.b[l][v], uv = u_in[v];
    u_out[v] = uv + w * (bv - stencil_apply<DIM, T>(L, v, c, u_in));
}

// Down the cycle on level l (not the last) from its right-hand side and first iterate:
// the other nu_pre - 1 Jacobi steps, the residual, its restriction to level l + 1. The
// iterate ends in u[nu_pre & 1].
template <int DIM, typename T, typename Each, typename Sync>
__device__ __forceinline__ void q1_down(const Q1Plan<T> &p, int l, bool last, const Each &each, Sync &sync) {
    const CGLevelDev<T> &L = p.L[l];
    T *u[2] = {p.u0[l], p.u1[l]};
    T *b = p.b[l], *r = p.r[l], *bn = p.b[l + 1];
    int c = p.nu_pre > 0 ? 1 : 0;
    for (int k = 1; k < p.nu_pre; ++k) {
        T *ui = u[c], *uo = u[c ^ 1];
        each(L.nv, [&](int64_t v) { q1_jacobi_at<DIM, T>(p, l, ui, uo, v); });
        c ^= 1;
        sync();
    }
    T *uc = u[c];
    each(L.nv, [&](int64_t v) { cg_residual_at<DIM, T>(L, uc, b, r, v); });
    sync();
    const int64_t ncv = DIM == 3 ? (int64_t)L.mc[0] * L.mc[1] * L.mc[2] : (int64_t)L.mc[0] * L.mc[1];
    each.warps(ncv * RS_LANES, [&](int64_t t) {   // whole warps: the lanes of a vertex exchange their sums
        const int64_t V = t / RS_LANES;
        const T s = h_restrict_at<DIM, T>(L, r, V < ncv ? V : -1);
        if (V >= ncv || t % RS_LANES != 0) return;
        if (last)
            bn[V] = s;
        else
            q1_put_rhs<T>(p, l + 1, V, s);
    });
    sync();
}

// Up the cycle on level l: add the prolongated correction ec of level l + 1,
// nu_post Jacobi steps; returns the level's result, u[(nu_pre + nu_post) & 1]. No
// barrier after the last step of level 0: the launch ends there.
template <int DIM, typename T, typename Each, typename Sync>
__device__ __forceinline__ const T *q1_up(const Q1Plan<T> &p, int l, const T *ec, const Each &each, Sync &sync) {
    const CGLevelDev<T> &L = p.L[l];
    T *u[2] = {p.u0[l], p.u1[l]};
    int c = p.nu_pre & 1;
    T *uc = u[c];
    each(L.nv, [&](int64_t v) { h_prolong_at<DIM, T>(L, ec, uc, v); });
    if (p.nu_post > 0 || l > 0) sync();
    for (int k = 0; k < p.nu_post; ++k) {
        T *ui = u[c], *uo = u[c ^ 1];
        each(L.nv, [&](int64_t v) { q1_jacobi_at<DIM, T>(p, l, ui, uo, v); });
        c ^= 1;
        if (k + 1 < p.nu_post || l > 0) sync();
    }
    return u[c];
}

// row i of e = E b, one warp: lane-strided (coalesced) products, four sums per lane
template <typename T>
__device__ __forceinline__ double q1_dense_row(int n, const double *__restrict__ E, const T *b, int64_t i) {
    const double *a = E + i * n;
    double s[4] = {};
    int j = threadIdx.x & 31;
    for (; j + 96 < n; j += 128)
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] = fma(__ldg(a + j + 32 * k), (double)b[j + 32 * k], s[k]);
    for (; j < n; j += 32) s[0] = fma(__ldg(a + j), (double)b[j], s[0]);
    double t = (s[0] + s[1]) + (s[2] + s[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

template <int DIM, typename T, int TPB>
__global__ void __launch_bounds__(TPB) k_q1_cycle(const __grid_constant__ Q1Plan<T> p,
                                                  const T *__restrict__ corners, unsigned long long *bar) {
    if (*(volatile unsigned long long *)&g_q1_barrier_timeouts != 0) return;
    // the finest level's stencil is first read after the first barrier: every block
    // requests its share into L2 now (a hint; 16-byte pieces)
    if (threadIdx.x == 0) {
        const uint64_t bytes = (uint64_t)(DIM == 3 ? 27 : 9) * p.L[0].nv * sizeof(T);
        const uint64_t chunk = ((bytes + gridDim.x - 1) / gridDim.x + 15) / 16 * 16;
        const uint64_t off = (uint64_t)blockIdx.x * chunk;
        const unsigned char *base = reinterpret_cast<const unsigned char *>(p.L[0].st);
        if (off < bytes && (reinterpret_cast<uintptr_t>(base) & 15) == 0) {
            const uint64_t n = (bytes - off < chunk ? bytes - off : chunk) / 16 * 16;
            if (n > 0)
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(base + off), "r"((unsigned)n)
                             : "memory");
        }
    }
    const int ld = p.dense_from;
    GridSync grid{bar, 0ull, 0u};
    const GridEach on_grid;
    on_grid(p.L[0].nv, [&](int64_t v) {
        q1_put_rhs<T>(p, 0, v, corner_sum_at<DIM, T>(p.L[0].m[0] + 1, p.L[0].m[1] + 1, p.L[0].m[2] + 1, corners, v));
    });
    grid();
    for (int l = 0; l < ld; ++l) q1_down<DIM, T>(p, l, l + 1 == ld, on_grid, grid);
    const T *bd = p.b[ld];
    T *e = p.u0[ld];
    const int nd = (int)p.ndense, warps = (int)gridDim.x * (TPB / 32);
    // consecutive warps of rows on different SMs
    for (int i = (int)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; i < nd; i += warps) {
        const double t = q1_dense_row<T>(nd, p.E, bd, i);
        if ((threadIdx.x & 31) == 0) e[i] = (T)t;
    }
    grid();
    const T *ec = e;
    for (int l = ld - 1; l >= 0; --l) ec = q1_up<DIM, T>(p, l, ec, on_grid, grid);
}

// The cycle of a problem whose level 0 is the dense one: every block gathers the
// right-hand side into shared memory, a warp per row.
template <int DIM, typename T>
__global__ void __launch_bounds__(Q1_TPB) k_q1_dense(const __grid_constant__ Q1Plan<T> p,
                                                     const T *__restrict__ corners) {
    extern __shared__ __align__(16) unsigned char q1_smem[];
    T *b = reinterpret_cast<T *>(q1_smem);
    const int n = (int)p.ndense;
    for (int v = threadIdx.x; v < n; v += blockDim.x)
        b[v] = corner_sum_at<DIM, T>(p.L[0].m[0] + 1, p.L[0].m[1] + 1, p.L[0].m[2] + 1, corners, v);
    __syncthreads();
    const int i = (int)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    if (i >= n) return;
    const double t = q1_dense_row<T>(n, p.E, b, i);
    if ((threadIdx.x & 31) == 0) p.u0[0][i] = (T)t;
}

// wd = omega / diagonal of the levels above the coarsest
template <int DIM, typename T>
__global__ void k_q1_weights(const __grid_constant__ Q1Plan<T> p, T omega) {
    for (int l = 0; l < p.nlev - 1; ++l)
        for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < p.L[l].nv; v += (int64_t)gridDim.x * blockDim.x)
            p.wd[l][v] = omega / p.L[l].st[(DIM == 3 ? 13 : 4) * p.L[l].nv + v];
}

// E[i][j]: the cycle from level dense_from down applied to the unit vectors e_j, one
// block per column, with the level vectors in shared memory. On level dense_from the
// iterates before the correction and the residual are zero beyond nu_pre vertices from
// j: those steps run on that box only (the FP64 pipe bounds the kernel: 1331 vertices
// 0.64 ms with all vertices in every step).
template <int DIM>
__global__ void __launch_bounds__(Q1_TPB) k_q1_dense_matrix(const __grid_constant__ Q1Plan<double> plan,
                                                            const double *__restrict__ Ainv, double *__restrict__ E) {
    extern __shared__ __align__(16) unsigned char q1_smem[];
    __shared__ Q1Plan<double> p;
    const int ld = plan.dense_from, nl = plan.nlev;
    if (threadIdx.x == 0) {
        p = plan;
        double *v = reinterpret_cast<double *>(q1_smem);
        for (int l = ld; l < nl; ++l) {
            const int64_t n = p.L[l].nv;
            p.u0[l] = v;
            p.u1[l] = v + n;
            p.b[l] = v + 2 * n;
            p.r[l] = v + 3 * n;
            v += 4 * n;
        }
    }
    __syncthreads();
    const BlockEach each;
    BlockSync sync;
    const CGLevelDev<double> &L = p.L[ld];
    const int64_t nd = L.nv, nc = p.L[nl - 1].nv, ncv = p.L[ld + 1].nv;
    const bool last = ld + 1 == nl - 1;
    double *u[2] = {p.u0[ld], p.u1[ld]}, *b = p.b[ld], *r = p.r[ld], *bn = p.b[ld + 1];
    for (int64_t j = blockIdx.x; j < nd; j += gridDim.x) {
        each(4 * nd, [&](int64_t v) { u[0][v] = 0.0; });   // u0, u1, b, r of the level
        sync();
        int cj[3] = {0, 0, 0};
        vcoords<DIM>(j, L.m, cj);
        // f(v) for the vertices at most `rad` from j
        auto box = [&](int rad, auto f) {
            int lo[3] = {0, 0, 0}, n[3] = {1, 1, 1};
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                lo[a] = max(cj[a] - rad, 0);
                n[a] = min(cj[a] + rad, L.m[a] - 1) - lo[a] + 1;
            }
            for (int k = threadIdx.x; k < n[0] * n[1] * n[2]; k += blockDim.x) {
                const int q = k / n[0], z = q / n[1];
                f((int64_t)(lo[0] + k - q * n[0]) + (int64_t)L.m[0] * ((lo[1] + q - z * n[1]) + (int64_t)L.m[1] * (lo[2] + z)));
            }
        };
        if (threadIdx.x == 0) q1_put_rhs<double>(p, ld, j, 1.0);
        sync();
        int c = p.nu_pre > 0 ? 1 : 0;
        for (int k = 1; k < p.nu_pre; ++k) {
            double *ui = u[c], *uo = u[c ^ 1];
            box(k, [&](int64_t v) { q1_jacobi_at<DIM, double>(p, ld, ui, uo, v); });
            c ^= 1;
            sync();
        }
        double *uc = u[c];
        box(p.nu_pre, [&](int64_t v) { cg_residual_at<DIM, double>(L, uc, b, r, v); });
        sync();
        each.warps(ncv * RS_LANES, [&](int64_t t) {
            const int64_t V = t / RS_LANES;
            const double s = h_restrict_at<DIM, double>(L, r, V < ncv ? V : -1);
            if (V >= ncv || t % RS_LANES != 0) return;
            if (last)
                bn[V] = s;
            else
                q1_put_rhs<double>(p, ld + 1, V, s);
        });
        sync();
        for (int l = ld + 1; l < nl - 1; ++l) q1_down<DIM, double>(p, l, l + 1 == nl - 1, each, sync);
        const double *rc = p.b[nl - 1];
        double *e = p.u0[nl - 1];
        each(nc, [&](int64_t i) { coarse_row<double>(nc, Ainv, rc, e, i); });
        sync();
        const double *ec = e;
        for (int l = nl - 2; l >= ld; --l) ec = q1_up<DIM, double>(p, l, ec, each, sync);
        sync();
        each(nd, [&](int64_t v) { E[v * nd + j] = ec[v]; });
        sync();
    }
}

// ---- batched forms: work item k covers vertices [v0, v0 + BATCH_VERTS) of
// descriptor map[k].desc (one level of one instance); all instances share one
// persistent launch per stage, whose CTAs stride through the nb work items.
template <int DIM, typename T>
__global__ void __launch_bounds__(BATCH_VERTS) k_corner_gather_batch(const BatchCG<T> *__restrict__ D,
                                                                     const VertMap *__restrict__ map, int nb) {
    for (int k = blockIdx.x; k < nb; k += gridDim.x) {
        const VertMap m = map[k];
        const BatchCG<T> &d = D[m.desc];
        corner_gather_at<DIM, T>(d.n[0], d.n[1], d.n[2], d.corners, d.b, (int64_t)m.v0 + threadIdx.x);
    }
}
template <int DIM, typename T>
__global__ void __launch_bounds__(BATCH_VERTS) k_cg_jacobi_batch(const BatchCG<T> *__restrict__ D,
                                                                 const VertMap *__restrict__ map, int nb, T omega,
                                                                 int zero_guess, int cur) {
    for (int k = blockIdx.x; k < nb; k += gridDim.x) {
        const VertMap m = map[k];
        const BatchCG<T> &d = D[m.desc];
        cg_jacobi_at<DIM, T>(d.L, d.u[cur], d.b, d.u[cur ^ 1], omega, zero_guess, (int64_t)m.v0 + threadIdx.x);
    }
}
template <int DIM, typename T>
__global__ void __launch_bounds__(BATCH_VERTS) k_cg_residual_batch(const BatchCG<T> *__restrict__ D,
                                                                   const VertMap *__restrict__ map, int nb, int cur) {
    for (int k = blockIdx.x; k < nb; k += gridDim.x) {
        const VertMap m = map[k];
        const BatchCG<T> &d = D[m.desc];
        cg_residual_at<DIM, T>(d.L, d.u[cur], d.b, d.r, (int64_t)m.v0 + threadIdx.x);
    }
}
template <int DIM, typename T>
__global__ void __launch_bounds__(BATCH_VERTS) k_h_restrict_batch(const BatchCG<T> *__restrict__ D,
                                                                  const VertMap *__restrict__ map, int nb) {
    for (int k = blockIdx.x; k < nb; k += gridDim.x) {
        const VertMap m = map[k];
        const BatchCG<T> &d = D[m.desc];
        const int64_t ncv = DIM == 3 ? (int64_t)d.L.mc[0] * d.L.mc[1] * d.L.mc[2] : (int64_t)d.L.mc[0] * d.L.mc[1];
        // the item's BATCH_VERTS vertices, RS_LANES threads each
        for (int64_t V = m.v0 + (int)threadIdx.x / RS_LANES, e = m.v0 + BATCH_VERTS; V < e; V += BATCH_VERTS / RS_LANES) {
            const T s = h_restrict_at<DIM, T>(d.L, d.r, V < ncv ? V : -1);
            if (V < ncv && threadIdx.x % RS_LANES == 0) d.b_next[V] = s;
        }
    }
}
template <int DIM, typename T>
__global__ void __launch_bounds__(BATCH_VERTS) k_h_prolong_batch(const BatchCG<T> *__restrict__ D,
                                                                 const VertMap *__restrict__ map, int nb, int cur) {
    for (int k = blockIdx.x; k < nb; k += gridDim.x) {
        const VertMap m = map[k];
        const BatchCG<T> &d = D[m.desc];
        h_prolong_at<DIM, T>(d.L, d.e_next, d.u[cur], (int64_t)m.v0 + threadIdx.x);
    }
}
template <typename T>
__global__ void __launch_bounds__(BATCH_VERTS) k_coarse_solve_batch(const BatchCG<T> *__restrict__ D,
                                                                    const VertMap *__restrict__ map, int nb) {
    for (int k = blockIdx.x; k < nb; k += gridDim.x) {
        const VertMap m = map[k];
        const BatchCG<T> &d = D[m.desc];
        coarse_row<T>(d.L.nv, d.Ainv, d.b, d.u[0], (int64_t)m.v0 + threadIdx.x);
    }
}

inline unsigned persistent_blocks(const void *fn, int threads, int nb) { return persistent_grid(fn, threads, 0, nb); }

inline unsigned blocks_for(int64_t n) { return (unsigned)((n + TPB - 1) / TPB); }

}  // namespace

// the kernel of precision T, dimension dim, 256 or (wide, FP32) 512 threads
template <typename T>
auto q1_cycle_fn(int dim, bool wide) -> void (*)(const Q1Plan<T>, const T *, unsigned long long *) {
    if constexpr (sizeof(T) == 4) {
        if (wide) return dim == 3 ? k_q1_cycle<3, T, Q1_TPB_WIDE> : k_q1_cycle<2, T, Q1_TPB_WIDE>;
    }
    return dim == 3 ? k_q1_cycle<3, T, Q1_TPB> : k_q1_cycle<2, T, Q1_TPB>;
}

template <typename T>
cudaError_t launch_q1_cycle(int dim, const Q1Plan<T> &plan, const T *corners, unsigned long long *bar, int blocks,
                            bool wide, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(wide && sizeof(T) == 4 ? Q1_TPB_WIDE : Q1_TPB);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // all blocks co-resident: the grid barrier cannot wait on an unscheduled block
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    count_launches(1);
    return cudaLaunchKernelEx(&cfg, q1_cycle_fn<T>(dim, wide), plan, corners, bar);
}

template <typename T>
cudaError_t launch_q1_dense(int dim, const Q1Plan<T> &plan, int64_t n, const T *corners, cudaStream_t s) {
    count_launches(1);
    const unsigned grid = (unsigned)((n + Q1_TPB / 32 - 1) / (Q1_TPB / 32));
    if (dim == 3)
        k_q1_dense<3, T><<<grid, Q1_TPB, n * sizeof(T), s>>>(plan, corners);
    else
        k_q1_dense<2, T><<<grid, Q1_TPB, n * sizeof(T), s>>>(plan, corners);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_q1_weights(int dim, const Q1Plan<T> &plan, T omega, cudaStream_t s) {
    count_launches(1);
    const unsigned grid = std::min(blocks_for(plan.L[0].nv), 1216u);
    if (dim == 3)
        k_q1_weights<3, T><<<grid, TPB, 0, s>>>(plan, omega);
    else
        k_q1_weights<2, T><<<grid, TPB, 0, s>>>(plan, omega);
    return cudaGetLastError();
}

// smem: bytes of the level vectors from dense_from down (4 per level)
cudaError_t launch_q1_dense_matrix(int dim, const Q1Plan<double> &plan, int64_t nd, size_t smem, const double *Ainv,
                                   double *E, cudaStream_t s) {
    count_launches(1);
    const auto fn = dim == 3 ? k_q1_dense_matrix<3> : k_q1_dense_matrix<2>;
    if (smem > 32 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Q1_DENSE_SMEM);
        if (e != cudaSuccess) return e;
    }
    fn<<<(unsigned)nd, Q1_TPB, smem, s>>>(plan, Ainv, E);
    return cudaGetLastError();
}

template <typename T>
int q1_cycle_max_blocks(int dim, bool wide) {
    int dev = 0, sms = 0, per = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    int coop = 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return 0;
    const int tpb = wide && sizeof(T) == 4 ? Q1_TPB_WIDE : Q1_TPB;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, q1_cycle_fn<T>(dim, wide), tpb, 0) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    // up to two blocks per SM: warps to hide the load latency of the vertex
    // loops; more would add arrivals at the grid barrier
    return per > 0 ? sms * (per < 2 ? per : 2) : 0;
}

cudaError_t q1_barrier_timeouts(unsigned long long *count) {
    return cudaMemcpyFromSymbol(count, g_q1_barrier_timeouts, sizeof(*count));
}
cudaError_t q1_barrier_timeouts_addr(unsigned long long **ptr) {
    return cudaGetSymbolAddress((void **)ptr, g_q1_barrier_timeouts);
}


template <typename T>
cudaError_t launch_corner_gather(int dim, const int *n, const T *corners, T *b0, cudaStream_t s) {
    const int64_t nv = dim == 3 ? (int64_t)(n[0] - 1) * (n[1] - 1) * (n[2] - 1) : (int64_t)(n[0] - 1) * (n[1] - 1);
    if (nv <= 0) return cudaSuccess;
    count_launches(1);
    if (dim == 3)
        k_corner_gather<3, T><<<blocks_for(nv), TPB, 0, s>>>(n[0], n[1], n[2], corners, b0);
    else
        k_corner_gather<2, T><<<blocks_for(nv), TPB, 0, s>>>(n[0], n[1], 1, corners, b0);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_cg_jacobi(int dim, const CGLevelDev<T> &L, const T *u_in, const T *b, T *u_out, T omega,
                             bool zero_guess, cudaStream_t s) {
    if (L.nv <= 0) return cudaSuccess;
    count_launches(1);
    if (dim == 3)
        k_cg_jacobi<3, T><<<blocks_for(L.nv), TPB, 0, s>>>(L, u_in, b, u_out, omega, zero_guess ? 1 : 0);
    else
        k_cg_jacobi<2, T><<<blocks_for(L.nv), TPB, 0, s>>>(L, u_in, b, u_out, omega, zero_guess ? 1 : 0);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_cg_residual(int dim, const CGLevelDev<T> &L, const T *u, const T *b, T *r, cudaStream_t s) {
    if (L.nv <= 0) return cudaSuccess;
    count_launches(1);
    if (dim == 3)
        k_cg_residual<3, T><<<blocks_for(L.nv), TPB, 0, s>>>(L, u, b, r);
    else
        k_cg_residual<2, T><<<blocks_for(L.nv), TPB, 0, s>>>(L, u, b, r);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_h_restrict(int dim, const CGLevelDev<T> &L, const T *rf, T *rc, cudaStream_t s) {
    const int64_t ncv = dim == 3 ? (int64_t)L.mc[0] * L.mc[1] * L.mc[2] : (int64_t)L.mc[0] * L.mc[1];
    if (ncv <= 0) return cudaSuccess;
    count_launches(1);
    if (dim == 3)
        k_h_restrict<3, T><<<blocks_for(ncv * RS_LANES), TPB, 0, s>>>(L, rf, rc);
    else
        k_h_restrict<2, T><<<blocks_for(ncv * RS_LANES), TPB, 0, s>>>(L, rf, rc);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_h_prolong(int dim, const CGLevelDev<T> &L, const T *ec, T *uf, cudaStream_t s) {
    if (L.nv <= 0) return cudaSuccess;
    count_launches(1);
    if (dim == 3)
        k_h_prolong<3, T><<<blocks_for(L.nv), TPB, 0, s>>>(L, ec, uf);
    else
        k_h_prolong<2, T><<<blocks_for(L.nv), TPB, 0, s>>>(L, ec, uf);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_coarse_solve(int64_t nc, const double *Ainv, const T *r, T *e, cudaStream_t s) {
    if (nc <= 0) return cudaSuccess;
    count_launches(1);
    k_coarse_solve<T><<<blocks_for(nc), TPB, 0, s>>>(nc, Ainv, r, e);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_corner_gather_batch(int dim, const BatchCG<T> *D, const VertMap *map, int nb, cudaStream_t s) {
    if (nb <= 0) return cudaSuccess;
    count_launches(1);
    if (dim == 3)
        k_corner_gather_batch<3, T><<<persistent_blocks((const void *)k_corner_gather_batch<3, T>, BATCH_VERTS, nb), BATCH_VERTS, 0, s>>>(D, map, nb);
    else
        k_corner_gather_batch<2, T><<<persistent_blocks((const void *)k_corner_gather_batch<2, T>, BATCH_VERTS, nb), BATCH_VERTS, 0, s>>>(D, map, nb);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_cg_jacobi_batch(int dim, const BatchCG<T> *D, const VertMap *map, int nb, T omega,
                                   bool zero_guess, int cur, cudaStream_t s) {
    if (nb <= 0) return cudaSuccess;
    count_launches(1);
    if (dim == 3)
        k_cg_jacobi_batch<3, T><<<persistent_blocks((const void *)k_cg_jacobi_batch<3, T>, BATCH_VERTS, nb), BATCH_VERTS, 0, s>>>(
            D, map, nb, omega, zero_guess ? 1 : 0, cur);
    else
        k_cg_jacobi_batch<2, T><<<persistent_blocks((const void *)k_cg_jacobi_batch<2, T>, BATCH_VERTS, nb), BATCH_VERTS, 0, s>>>(
            D, map, nb, omega, zero_guess ? 1 : 0, cur);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_cg_residual_batch(int dim, const BatchCG<T> *D, const VertMap *map, int nb, int cur,
                                     cudaStream_t s) {
    if (nb <= 0) return cudaSuccess;
    count_launches(1);
    if (dim == 3)
        k_cg_residual_batch<3, T><<<persistent_blocks((const void *)k_cg_residual_batch<3, T>, BATCH_VERTS, nb), BATCH_VERTS, 0, s>>>(
            D, map, nb, cur);
    else
        k_cg_residual_batch<2, T><<<persistent_blocks((const void *)k_cg_residual_batch<2, T>, BATCH_VERTS, nb), BATCH_VERTS, 0, s>>>(
            D, map, nb, cur);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_h_restrict_batch(int dim, const BatchCG<T> *D, const VertMap *map, int nb, cudaStream_t s) {
    if (nb <= 0) return cudaSuccess;
    count_launches(1);
    if (dim == 3)
        k_h_restrict_batch<3, T><<<persistent_blocks((const void *)k_h_restrict_batch<3, T>, BATCH_VERTS, nb), BATCH_VERTS, 0, s>>>(
            D, map, nb);
    else
        k_h_restrict_batch<2, T><<<persistent_blocks((const void *)k_h_restrict_batch<2, T>, BATCH_VERTS, nb), BATCH_VERTS, 0, s>>>(
            D, map, nb);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_h_prolong_batch(int dim, const BatchCG<T> *D, const VertMap *map, int nb, int cur,
                                   cudaStream_t s) {
    if (nb <= 0) return cudaSuccess;
    count_launches(1);
    if (dim == 3)
        k_h_prolong_batch<3, T><<<persistent_blocks((const void *)k_h_prolong_batch<3, T>, BATCH_VERTS, nb), BATCH_VERTS, 0, s>>>(
            D, map, nb, cur);
    else
        k_h_prolong_batch<2, T><<<persistent_blocks((const void *)k_h_prolong_batch<2, T>, BATCH_VERTS, nb), BATCH_VERTS, 0, s>>>(
            D, map, nb, cur);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_coarse_solve_batch(const BatchCG<T> *D, const VertMap *map, int nb, cudaStream_t s) {
    if (nb <= 0) return cudaSuccess;
    count_launches(1);
    k_coarse_solve_batch<T><<<persistent_blocks((const void *)k_coarse_solve_batch<T>, BATCH_VERTS, nb), BATCH_VERTS, 0, s>>>(D, map, nb);
    return cudaGetLastError();
}

#define DGMG_CG_INST(T)                                                                                         \
    template cudaError_t launch_corner_gather<T>(int, const int *, const T *, T *, cudaStream_t);              \
    template cudaError_t launch_cg_jacobi<T>(int, const CGLevelDev<T> &, const T *, const T *, T *, T, bool,   \
                                             cudaStream_t);                                                    \
    template cudaError_t launch_cg_residual<T>(int, const CGLevelDev<T> &, const T *, const T *, T *,          \
                                               cudaStream_t);                                                  \
    template cudaError_t launch_h_restrict<T>(int, const CGLevelDev<T> &, const T *, T *, cudaStream_t);       \
    template cudaError_t launch_h_prolong<T>(int, const CGLevelDev<T> &, const T *, T *, cudaStream_t);        \
    template cudaError_t launch_coarse_solve<T>(int64_t, const double *, const T *, T *, cudaStream_t);        \
    template cudaError_t launch_corner_gather_batch<T>(int, const BatchCG<T> *, const VertMap *, int,           \
                                                       cudaStream_t);                                          \
    template cudaError_t launch_cg_jacobi_batch<T>(int, const BatchCG<T> *, const VertMap *, int, T, bool, int, \
                                                   cudaStream_t);                                              \
    template cudaError_t launch_cg_residual_batch<T>(int, const BatchCG<T> *, const VertMap *, int, int,         \
                                                     cudaStream_t);                                            \
    template cudaError_t launch_h_restrict_batch<T>(int, const BatchCG<T> *, const VertMap *, int, cudaStream_t); \
    template cudaError_t launch_h_prolong_batch<T>(int, const BatchCG<T> *, const VertMap *, int, int,          \
                                                   cudaStream_t);                                              \
    template cudaError_t launch_coarse_solve_batch<T>(const BatchCG<T> *, const VertMap *, int, cudaStream_t);

DGMG_CG_INST(double)
DGMG_CG_INST(float)

#define DGMG_Q1_INST(T)                                                                                               \
    template cudaError_t launch_q1_cycle<T>(int, const Q1Plan<T> &, const T *, unsigned long long *, int, bool,        \
                                            cudaStream_t);                                                            \
    template cudaError_t launch_q1_dense<T>(int, const Q1Plan<T> &, int64_t, const T *, cudaStream_t);                 \
    template cudaError_t launch_q1_weights<T>(int, const Q1Plan<T> &, T, cudaStream_t);
DGMG_Q1_INST(double)
DGMG_Q1_INST(float)
template int q1_cycle_max_blocks<double>(int, bool);
template int q1_cycle_max_blocks<float>(int, bool);

}  // namespace dgmg
