// Vector kernels of the outer conjugate-gradient loop, FP64 and FP32: deterministic
// dot products (grid a function of the length, fixed reduction order), the CG updates
// with step lengths read from device memory, precision casts, and the
// right-hand-side quadrature (b_i = (f, phi_i), the right-hand side of
// Eq. weak_form_IP). The CG loop uses one multigrid cycle as its preconditioner
// (P^-1 of Sec. 5.1 "Exit criterion").
#include <algorithm>
#include <type_traits>

#include "internal.h"

namespace dgmg {

namespace {

// the block's W sums of s in thread 0, in a fixed order
template <int W>
__device__ __forceinline__ void block_sums(const double *s, double *v, double (*sh)[32]) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
        double t = s[w];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if ((threadIdx.x & 31) == 0) sh[w][threadIdx.x >> 5] = t;
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < W; ++w) {
        v[w] = 0.0;
        if (threadIdx.x < 32) {
            v[w] = threadIdx.x < (blockDim.x >> 5) ? sh[w][threadIdx.x] : 0.0;
            for (int o = 16; o > 0; o >>= 1) v[w] += __shfl_down_sync(0xffffffffu, v[w], o);
        }
    }
}

// One vector load of 16 bytes, or (VEC = false: some vector is not 16-byte aligned)
// one element.
template <typename T, bool VEC>
struct Pack {
    static constexpr int N = VEC ? 16 / (int)sizeof(T) : 1;
    alignas(VEC ? 16 : sizeof(T)) T v[N];
    __device__ __forceinline__ void load(const T *p) {
        if constexpr (VEC) {
            using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
            *reinterpret_cast<V *>(v) = *reinterpret_cast<const V *>(p);
        } else {
            v[0] = *p;
        }
    }
    __device__ __forceinline__ void store(T *p) const {
        if constexpr (VEC) {
            using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
            *reinterpret_cast<V *>(p) = *reinterpret_cast<const V *>(v);
        } else {
            *p = v[0];
        }
    }
};

// s += a.b of two packs, accumulated in FP64. FP32: the four products of a pack are
// summed in FP32 (fused multiply-adds) first; such a group sum carries an error of a
// few FP32 ulps of its terms, the order of the rounding of the vector entries
// themselves. Single elements are multiplied in FP64. (The group sums widened by the
// FP64 pipe bound two products of 32.8M values: 129 us, where memory takes 58.)
template <typename T, bool VEC>
__device__ __forceinline__ void pack_dot(double &s, const Pack<T, VEC> &a, const Pack<T, VEC> &b) {
    if constexpr (VEC && sizeof(T) == 4) {
        s += widen(fmaf(a.v[3], b.v[3], fmaf(a.v[2], b.v[2], fmaf(a.v[1], b.v[1], a.v[0] * b.v[0]))));
    } else {
#pragma unroll
        for (int e = 0; e < Pack<T, VEC>::N; ++e) s = fma((double)a.v[e], (double)b.v[e], s);
    }
}

// The end of a dot product: every block stores its W partial sums; the block that
// arrives last at the ticket (which wraps back to 0) adds them up in their fixed order
// and writes out[0 .. W). One launch instead of two (a second kernel costs 3.7 us and
// a launch gap). scal, when given: the CG direction update's beta from <r,z> = out[0]
// (Fletcher-Reeves; with W = 2 Polak-Ribiere, out[1] = <r_old,z>) and the shift of <r,z>.
template <int W>
__device__ __forceinline__ void dot_finish(const double *s, double *partials, double *out0, double *out1, double *scal) {
    __shared__ double sh[W][32];
    __shared__ unsigned last;
    double v[W];
    block_sums<W>(s, v, sh);
    if (threadIdx.x == 0)
#pragma unroll
        for (int w = 0; w < W; ++w) partials[w * DOT_BLOCKS + blockIdx.x] = v[w];
    unsigned *ticket = reinterpret_cast<unsigned *>(partials + 2 * DOT_BLOCKS);
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double t[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
        t[w] = 0.0;
        for (unsigned i = threadIdx.x; i < gridDim.x; i += blockDim.x) t[w] += __ldcg(partials + w * DOT_BLOCKS + i);
    }
    block_sums<W>(t, v, sh);
    if (threadIdx.x == 0) {
        if (out0) *out0 = v[0];
        if (W == 2 && out1) *out1 = v[W - 1];
        if (scal) {
            scal[2] = W == 2 ? (v[0] - v[W - 1]) / scal[0] : v[0] / scal[0];   // beta
            scal[0] = v[0];                                                   // <r,z>
        }
    }
}

// out0 = a.b, and with W = 2 out1 = c.b (b read once). Four loads per vector in flight.
template <typename T, int W, bool VEC>
__global__ void __launch_bounds__(DOT_THREADS, 4) k_dot(int64_t n, const T *__restrict__ a, const T *__restrict__ b,
                                                     const T *__restrict__ c, double *__restrict__ partials, double *out0,
                                                     double *out1, double *scal) {
    using P = Pack<T, VEC>;
    constexpr int U = 4;
    const int64_t nv = n / P::N, stride = (int64_t)gridDim.x * blockDim.x;
    double s[W] = {}, t[W] = {};
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + (U - 1) * stride < nv; i += U * stride) {
        P x[U], y[U], z[W == 2 ? U : 1];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            y[k].load(b + (i + k * stride) * P::N);
            x[k].load(a + (i + k * stride) * P::N);
            if constexpr (W == 2) z[k].load(c + (i + k * stride) * P::N);
        }
#pragma unroll
        for (int k = 0; k < U; ++k) {
            pack_dot<T, VEC>(k & 1 ? t[0] : s[0], x[k], y[k]);
            if constexpr (W == 2) pack_dot<T, VEC>(k & 1 ? t[1] : s[1], z[k], y[k]);
        }
    }
    for (; i < nv; i += stride) {
        P x, y;
        y.load(b + i * P::N);
        x.load(a + i * P::N);
        pack_dot<T, VEC>(s[0], x, y);
        if constexpr (W == 2) {
            x.load(c + i * P::N);
            pack_dot<T, VEC>(s[1], x, y);
        }
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1)
        for (int64_t k = nv * P::N; k < n; ++k) {
            s[0] = fma((double)a[k], (double)b[k], s[0]);
            if constexpr (W == 2) s[1] = fma((double)c[k], (double)b[k], s[1]);
        }
#pragma unroll
    for (int w = 0; w < W; ++w) s[w] += t[w];
    dot_finish<W>(s, partials, out0, out1, scal);
}

// out0 = ||r||^2, out1 = ||x - y||^2 (the two norms of a stationary iteration)
template <bool VEC>
__global__ void __launch_bounds__(DOT_THREADS) k_norms(int64_t n, const double *__restrict__ r, const double *__restrict__ x,
                                                       const double *__restrict__ y, double *__restrict__ partials,
                                                       double *out0, double *out1) {
    using P = Pack<double, VEC>;
    const int64_t nv = n / P::N, stride = (int64_t)gridDim.x * blockDim.x;
    double s[2] = {};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += stride) {
        P a, b, c;
        a.load(r + i * P::N);
        b.load(x + i * P::N);
        c.load(y + i * P::N);
        pack_dot<double, VEC>(s[0], a, a);
#pragma unroll
        for (int e = 0; e < P::N; ++e) b.v[e] -= c.v[e];
        pack_dot<double, VEC>(s[1], b, b);
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1)
        for (int64_t k = nv * P::N; k < n; ++k) {
            const double d = x[k] - y[k];
            s[0] = fma(r[k], r[k], s[0]);
            s[1] = fma(d, d, s[1]);
        }
    dot_finish<2>(s, partials, out0, out1, nullptr);
}

// x += alpha p, r_old = r (when given), r -= alpha q, out = ||r||^2 of the new r in the
// same pass; alpha = scal[0] / scal[1] = <r,z> / <p,q>
template <typename T, bool VEC>
__global__ void __launch_bounds__(DOT_THREADS) k_update_xr(int64_t n, T *__restrict__ x, T *__restrict__ r,
                                                           T *__restrict__ rold, const T *__restrict__ p,
                                                           const T *__restrict__ q, const double *__restrict__ scal,
                                                           double *__restrict__ partials, double *out) {
    using P = Pack<T, VEC>;
    const T alpha = (T)(scal[0] / scal[1]);
    const int64_t nv = n / P::N, stride = (int64_t)gridDim.x * blockDim.x;
    double s[1] = {};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += stride) {
        P ri, pi, qi, xi;
        ri.load(r + i * P::N);
        pi.load(p + i * P::N);
        qi.load(q + i * P::N);
        xi.load(x + i * P::N);
        if (rold) ri.store(rold + i * P::N);
#pragma unroll
        for (int e = 0; e < P::N; ++e) {
            xi.v[e] = fma(alpha, pi.v[e], xi.v[e]);
            ri.v[e] = fma(-alpha, qi.v[e], ri.v[e]);
        }
        xi.store(x + i * P::N);
        ri.store(r + i * P::N);
        pack_dot<T, VEC>(s[0], ri, ri);
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1)
        for (int64_t k = nv * P::N; k < n; ++k) {
            const T ri = r[k], rn = fma(-alpha, q[k], ri);
            if (rold) rold[k] = ri;
            x[k] = fma(alpha, p[k], x[k]);
            r[k] = rn;
            s[0] = fma((double)rn, (double)rn, s[0]);
        }
    dot_finish<1>(s, partials, out, nullptr, nullptr);
}

// p = z + beta p, beta = scal[2]
template <typename T, bool VEC>
__global__ void __launch_bounds__(DOT_THREADS) k_update_p(int64_t n, T *__restrict__ p, const T *__restrict__ z,
                                                          const double *__restrict__ scal) {
    using P = Pack<T, VEC>;
    const T beta = (T)scal[2];
    const int64_t nv = n / P::N, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += stride) {
        P pi, zi;
        pi.load(p + i * P::N);
        zi.load(z + i * P::N);
#pragma unroll
        for (int e = 0; e < P::N; ++e) pi.v[e] = fma(beta, pi.v[e], zi.v[e]);
        pi.store(p + i * P::N);
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1)
        for (int64_t k = nv * P::N; k < n; ++k) p[k] = fma(beta, p[k], z[k]);
}

__global__ void k_d2f(int64_t n, const double *__restrict__ x, float *__restrict__ y) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = (float)x[i];
}

__global__ void k_f2d(int64_t n, const float *__restrict__ x, double *__restrict__ y) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = (double)x[i];
}

// x += xs (FP64 accumulation of the FP32 correction), xs = 0
__global__ void k_accumulate_f2d(int64_t n, double *__restrict__ x, float *__restrict__ xs) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        x[i] += (double)xs[i];
        xs[i] = 0.0f;
    }
}


// physical coordinates of the mq^d Gauss points of every cell
__global__ void k_quad_points(int dim, int n0, int n1, int n2, int mq, const double *__restrict__ xq1,
                              double *__restrict__ xq, int64_t ncell) {
    const int64_t npc = dim == 3 ? (int64_t)mq * mq * mq : (int64_t)mq * mq;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= ncell * npc) return;
    const int64_t cell = idx / npc;
    const int g = (int)(idx % npc);
    const int gi[3] = {g % mq, (g / mq) % mq, g / (mq * mq)};
    const int ci[3] = {(int)(cell % n0), (int)((cell / n0) % n1), (int)(cell / ((int64_t)n0 * n1))};
    const int n[3] = {n0, n1, n2};
    for (int a = 0; a < dim; ++a) xq[idx * dim + a] = (ci[a] + 0.5 * (xq1[gi[a]] + 1.0)) / n[a];
}

// b[cell][node] = sum_g w_g f_g phi_node(x_g) with phi = product of 1D Lagrange
// values V[i][g] (q x mq) and w = product of the 1D Gauss weights scaled to the
// cell, sum-factorised: one CTA per cell contracts the mq^d point values with
// W_a[i][g] = V[i][g] w_a[g] one axis at a time (x, then y, then z).
constexpr int LV_THREADS = 128;
constexpr int LV_MQ = QMAX + 1;     // Gauss points per axis of the load quadrature (p + 2)
__global__ void __launch_bounds__(LV_THREADS) k_load_vector(int dim, int q, int mq, int64_t ncell,
                                                            const double *__restrict__ V,
                                                            const double *__restrict__ wq,
                                                            const double *__restrict__ fq, double *__restrict__ b) {
    __shared__ double sW[3][QMAX * LV_MQ];
    __shared__ double sF[LV_MQ * LV_MQ * LV_MQ];
    __shared__ double s1[QMAX * LV_MQ * LV_MQ];
    __shared__ double s2[QMAX * QMAX * LV_MQ];
    const int64_t cell = blockIdx.x;
    const int t = threadIdx.x;
    const int npc = dim == 3 ? mq * mq * mq : mq * mq;
    for (int e = t; e < dim * q * mq; e += blockDim.x) {
        const int a = e / (q * mq), r = e - a * q * mq, g = r % mq;
        sW[a][r] = V[r] * wq[a * mq + g];
    }
    for (int e = t; e < npc; e += blockDim.x) sF[e] = fq[cell * npc + e];
    __syncthreads();
    // x: s1[i + q (g2 + mq g3)] = sum_g1 W_x[i][g1] f[g1 + mq (g2 + mq g3)]
    const int n1 = dim == 3 ? q * mq * mq : q * mq;
    for (int e = t; e < n1; e += blockDim.x) {
        const int i = e % q, rest = e / q;
        double s = 0.0;
        for (int g = 0; g < mq; ++g) s = fma(sW[0][i * mq + g], sF[g + mq * rest], s);
        s1[e] = s;
    }
    __syncthreads();
    const int nl = dim == 3 ? q * q * q : q * q;
    double *out = b + cell * nl;
    if (dim == 2) {
        // y: b[i + q j] = sum_g2 W_y[j][g2] s1[i + q g2]
        for (int e = t; e < nl; e += blockDim.x) {
            const int i = e % q, j = e / q;
            double s = 0.0;
            for (int g = 0; g < mq; ++g) s = fma(sW[1][j * mq + g], s1[i + q * g], s);
            out[e] = s;
        }
        return;
    }
    // y: s2[i + q (j + q g3)] = sum_g2 W_y[j][g2] s1[i + q (g2 + mq g3)]
    const int n2 = q * q * mq;
    for (int e = t; e < n2; e += blockDim.x) {
        const int i = e % q, j = (e / q) % q, g3 = e / (q * q);
        double s = 0.0;
        for (int g = 0; g < mq; ++g) s = fma(sW[1][j * mq + g], s1[i + q * (g + mq * g3)], s);
        s2[e] = s;
    }
    __syncthreads();
    // z: b[i + q (j + q k)] = sum_g3 W_z[k][g3] s2[i + q (j + q g3)]
    for (int e = t; e < nl; e += blockDim.x) {
        const int ij = e % (q * q), k = e / (q * q);
        double s = 0.0;
        for (int g = 0; g < mq; ++g) s = fma(sW[2][k * mq + g], s2[ij + q * q * g], s);
        out[e] = s;
    }
}

inline unsigned grid_for(int64_t n) {
    const int64_t b = (n + 255) / 256;
    return (unsigned)(b < 4 * 152 * 4 ? (b > 0 ? b : 1) : 4 * 152 * 4);
}

}  // namespace

inline bool aligned16(const void *a, const void *b, const void *c = nullptr, const void *d = nullptr,
                      const void *e = nullptr) {
    return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(c) |
             reinterpret_cast<uintptr_t>(d) | reinterpret_cast<uintptr_t>(e)) & 15) == 0;
}

// blocks of a vector kernel: about two rounds of 16-byte loads per thread, at most four
// blocks per SM; a function of the length alone, so the sums have one order per length
static unsigned vector_blocks(int64_t n, int item) {
    const int64_t b = (n * item / 16 + 2 * DOT_THREADS - 1) / (2 * DOT_THREADS);
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(b, DOT_BLOCKS));
}

template <typename T>
cudaError_t launch_dot(int64_t n, const T *a, const T *b, double *partials, double *out, cudaStream_t s, double *scal) {
    count_launches(1);
    const unsigned g = vector_blocks(n, sizeof(T));
    if (aligned16(a, b))
        k_dot<T, 1, true><<<g, DOT_THREADS, 0, s>>>(n, a, b, nullptr, partials, out, nullptr, scal);
    else
        k_dot<T, 1, false><<<g, DOT_THREADS, 0, s>>>(n, a, b, nullptr, partials, out, nullptr, scal);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_dot2(int64_t n, const T *a, const T *b, const T *c, double *partials, double *out_ab, double *out_cb,
                        cudaStream_t s, double *scal) {
    count_launches(1);
    const unsigned g = vector_blocks(n, sizeof(T));
    if (aligned16(a, b, c))
        k_dot<T, 2, true><<<g, DOT_THREADS, 0, s>>>(n, a, b, c, partials, out_ab, out_cb, scal);
    else
        k_dot<T, 2, false><<<g, DOT_THREADS, 0, s>>>(n, a, b, c, partials, out_ab, out_cb, scal);
    return cudaGetLastError();
}
cudaError_t launch_norms(int64_t n, const double *r, const double *x, const double *y, double *partials, double *out_rr,
                         double *out_dd, cudaStream_t s) {
    count_launches(1);
    const unsigned g = vector_blocks(n, sizeof(double));
    if (aligned16(r, x, y))
        k_norms<true><<<g, DOT_THREADS, 0, s>>>(n, r, x, y, partials, out_rr, out_dd);
    else
        k_norms<false><<<g, DOT_THREADS, 0, s>>>(n, r, x, y, partials, out_rr, out_dd);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_update_xr(int64_t n, T *x, T *r, T *rold, const T *p, const T *q, const double *scal,
                             double *partials, double *out_rr, cudaStream_t s) {
    count_launches(1);
    const unsigned g = vector_blocks(n, sizeof(T));
    if (aligned16(x, r, rold, p, q))
        k_update_xr<T, true><<<g, DOT_THREADS, 0, s>>>(n, x, r, rold, p, q, scal, partials, out_rr);
    else
        k_update_xr<T, false><<<g, DOT_THREADS, 0, s>>>(n, x, r, rold, p, q, scal, partials, out_rr);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_update_p(int64_t n, T *p, const T *z, const double *scal, cudaStream_t s) {
    count_launches(1);
    const unsigned g = vector_blocks(n, sizeof(T));
    if (aligned16(p, z))
        k_update_p<T, true><<<g, DOT_THREADS, 0, s>>>(n, p, z, scal);
    else
        k_update_p<T, false><<<g, DOT_THREADS, 0, s>>>(n, p, z, scal);
    return cudaGetLastError();
}
#define DGMG_BLAS_INST(T)                                                                                             \
    template cudaError_t launch_dot<T>(int64_t, const T *, const T *, double *, double *, cudaStream_t, double *);     \
    template cudaError_t launch_dot2<T>(int64_t, const T *, const T *, const T *, double *, double *, double *,        \
                                        cudaStream_t, double *);                                                      \
    template cudaError_t launch_update_xr<T>(int64_t, T *, T *, T *, const T *, const T *, const double *, double *,   \
                                             double *, cudaStream_t);                                                 \
    template cudaError_t launch_update_p<T>(int64_t, T *, const T *, const double *, cudaStream_t);
DGMG_BLAS_INST(double)
DGMG_BLAS_INST(float)

cudaError_t launch_cast_d2f(int64_t n, const double *x, float *y, cudaStream_t s) {
    count_launches(1);
    k_d2f<<<grid_for(n), 256, 0, s>>>(n, x, y);
    return cudaGetLastError();
}

cudaError_t launch_cast_f2d(int64_t n, const float *x, double *y, cudaStream_t s) {
    count_launches(1);
    k_f2d<<<grid_for(n), 256, 0, s>>>(n, x, y);
    return cudaGetLastError();
}

cudaError_t launch_quad_points(int dim, int q, const int *n, int mq, const double *xq1, double *xq, int64_t ncell,
                               cudaStream_t s) {
    (void)q;
    const int64_t npc = dim == 3 ? (int64_t)mq * mq * mq : (int64_t)mq * mq;
    const int64_t tot = ncell * npc;
    if (tot == 0) return cudaSuccess;
    count_launches(1);
    k_quad_points<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(dim, n[0], n[1], dim == 3 ? n[2] : 1, mq, xq1, xq,
                                                                 ncell);
    return cudaGetLastError();
}

cudaError_t launch_load_vector(int dim, int q, int mq, int64_t ncell, const double *V, const double *wq,
                               const double *fq, double *b, cudaStream_t s) {
    const int64_t nl = dim == 3 ? (int64_t)q * q * q : (int64_t)q * q;
    const int64_t tot = ncell * nl;
    if (tot == 0) return cudaSuccess;
    if (q > QMAX || mq > LV_MQ || ncell > 0x7fffffff) return cudaErrorInvalidValue;
    count_launches(1);
    k_load_vector<<<(unsigned)ncell, LV_THREADS, 0, s>>>(dim, q, mq, ncell, V, wq, fq, b);
    return cudaGetLastError();
}

cudaError_t launch_accumulate_f2d(int64_t n, double *x, float *xs, cudaStream_t s) {
    count_launches(1);
    k_accumulate_f2d<<<grid_for(n), 256, 0, s>>>(n, x, xs);
    return cudaGetLastError();
}


// ---------------------------------------------------------------- FMA peak
// Every thread runs CH independent chains of fused multiply-adds (x <- x a + b,
// |a| < 1, so the values stay bounded); the chains' sum is stored only if it
// equals a value it cannot reach, which keeps the work live without a store.
__device__ double g_fma_sink;   // external linkage: the store cannot be dropped

// Register operands only: a and b pass through an opaque move per chain, so the
// multiply-add reads no constant-bank operand.
__device__ __forceinline__ double opaque(double v) {
    double r;
    asm volatile("mov.b64 %0, %1;" : "=d"(r) : "d"(v));
    return r;
}
__device__ __forceinline__ float opaque(float v) {
    float r;
    asm volatile("mov.b32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

template <typename T, int CH>
__global__ void __launch_bounds__(256) k_fma_loop(int iters, T a, T b) {
    T x[CH], ac[CH], bc[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        x[c] = (T)(threadIdx.x + c) * (T)1e-3;
        ac[c] = opaque(a);
        bc[c] = opaque(b);
    }
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int c = 0; c < CH; ++c) x[c] = fma(x[c], ac[c], bc[c]);
    }
    T s = T(0);
#pragma unroll
    for (int c = 0; c < CH; ++c) s += x[c];
    if (s == (T)-1.0) g_fma_sink = (double)s;
}

// The same on packed pairs: one instruction updates two lanes of a float2.
template <int CH>
__global__ void __launch_bounds__(256) k_fma_loop_x2(int iters, float a, float b) {
    float2 x[CH];
    const float2 a2 = make_float2(opaque(a), opaque(a)), b2 = make_float2(opaque(b), opaque(b));
#pragma unroll
    for (int c = 0; c < CH; ++c) x[c] = make_float2((threadIdx.x + c) * 1e-3f, (threadIdx.x + c) * 2e-3f);
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int c = 0; c < CH; ++c) x[c] = __ffma2_rn(x[c], a2, b2);
    }
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < CH; ++c) s += x[c].x + x[c].y;
    if (s == -1.f) g_fma_sink = (double)s;
}

}  // namespace dgmg

extern "C" int dgmg_fma_peak(int kind, double *tflops, void *stream) {
    using namespace dgmg;
    if (!tflops) return fail(DGMG_EINVAL, "dgmg_fma_peak: tflops is NULL");
    if (kind < 0 || kind > 2) return fail(DGMG_EINVAL, "dgmg_fma_peak: kind must be 0, 1 or 2");
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0, sms = 0, per = 0;
    DG_CUDA(cudaGetDevice(&dev));
    DG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    constexpr int CH = 8, TPB = 256;
    if (kind == 0)
        DG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_fma_loop<double, CH>, TPB, 0));
    else if (kind == 1)
        DG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_fma_loop<float, CH>, TPB, 0));
    else
        DG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_fma_loop_x2<CH>, TPB, 0));
    per = per > 0 ? per : 1;
    const double lanes = kind == 2 ? 2.0 : 1.0;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    DG_CUDA(cudaEventCreate(&e0));
    DG_CUDA(cudaEventCreate(&e1));
    auto run = [&](int blocks, int iters) -> cudaError_t {
        count_launches(1);
        if (kind == 0)
            k_fma_loop<double, CH><<<blocks, TPB, 0, s>>>(iters, 0.999999, 1e-7);
        else if (kind == 1)
            k_fma_loop<float, CH><<<blocks, TPB, 0, s>>>(iters, 0.9999f, 1e-4f);
        else
            k_fma_loop_x2<CH><<<blocks, TPB, 0, s>>>(iters, 0.9999f, 1e-4f);
        return cudaGetLastError();
    };
    // resident blocks per SM from one to the occupancy limit; per shape the
    // iterations are calibrated to about 30 ms, then the best of three timed
    // launches is kept; the best shape gives the peak
    double best_rate = 0.0;
    cudaError_t e = cudaSuccess;
    int shapes[16], nshape = 0;
    for (int b = 1; b < per && nshape < 15; b *= 2) shapes[nshape++] = b;
    shapes[nshape++] = per;
    for (int si = 0; si < nshape && e == cudaSuccess; ++si) {
        const int blocks = sms * shapes[si];
        int iters = kind == 0 ? 64 : 2048;
        float ms = 0.f, best = 0.f;
        e = run(blocks, iters);   // warm-up
        for (int k = 0; k < 6 && e == cudaSuccess; ++k) {
            e = cudaEventRecord(e0, s);
            if (e == cudaSuccess) e = run(blocks, iters);
            if (e == cudaSuccess) e = cudaEventRecord(e1, s);
            if (e == cudaSuccess) e = cudaEventSynchronize(e1);
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
            if (e != cudaSuccess) break;
            if (k < 3) {
                if (ms < 30.f)
                    iters = (int)std::min<double>(iters * std::max(2.0, 30.0 / std::max(ms, 0.01f)), 1 << 26);
                continue;
            }
            if (best == 0.f || ms < best) best = ms;
        }
        if (e == cudaSuccess && best > 0.f) {
            const double fmas = (double)blocks * TPB * CH * 4.0 * iters * lanes;
            best_rate = std::max(best_rate, 2.0 * fmas / (best * 1e-3) / 1e12);
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (e != cudaSuccess) return cuda_fail(e, "dgmg_fma_peak");
    *tflops = best_rate;
    return DGMG_OK;
}
