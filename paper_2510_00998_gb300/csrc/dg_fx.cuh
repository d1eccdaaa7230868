// FP64 kernels of the DG levels in block fixed-point arithmetic (fx.cuh): warm-up
// projection, smoothing step, residual. 2D and 3D, every degree, both bases, exact
// and interior-only blocks.
//
// Work decomposition. q lanes of a warp serve one cell (32 / q cells per warp; small 3D
// meshes of q >= 5: SP lanes per slab, fx_split); the
// cell tensor stays in shared memory as 64-bit integers of one exponent per cell. A
// pass along an axis takes the cell's q^(d-1) pencils, q^(d-2) per lane: load q
// values, apply a q x q matrix held in registers, store. Lane k's pencils along the
// first axes lie in its own slab (3D: the plane z = k, 2D: the row y = k), those
// along the last axis cross the slabs, so a warp barrier is all that separates two
// passes, and no CTA barrier follows the staging of the tables. The loops over
// pencils and axes stay rolled: one copy of each pass serves all axes (unrolled, the
// q = 4 step is 10,000 instructions that every warp runs once, more than the
// instruction cache holds, at 168 to 255 registers; rolled it takes half of them,
// and every degree fits).
//
// Facet terms without facet masses. With M = Mx (x) My (x) Mz the facet terms of
// axis a are M (n (x) f): the tangential masses applied to the neighbour's trace f
// are those of M, and along the axis M_a times n = M_a^-1 (end vector). So the
// kernels add, per axis, the rank-four update n (x) f of the neighbours' traces
// (and, in the residual, D_a u with D_a = M_a^-1 Kt_a, the cell's own 1D block)
// pencil by pencil, and apply M once to the sum over the axes:
//   A u = M [ sum_a D_a u + sum_faces n (x) f ],
// d q multiply-adds per node for M instead of two tangential masses per face and
// field, and no mass at all in the first step from a zero iterate.
//
// Numbers: a pass rounds to the block's unit, node-wise sums with the caller's vectors (b, u)
// are FP64 (their pipe is idle otherwise: 5% busy).
//
// What bounds it: the integer multiply-add pipe (57% busy at q = 4 with a last wave of
// CTAs that fills 68% of the chip; about 290 of its instructions per node of a smoothing
// step) with the ALU at 28% and 12 to 16 warps per SM to cover the latencies. Measured
// per launch, FP64 pipe kernels before / these: smoothing step 33 x 31 x 32 cells
// p = 3 0.261 / 0.093 ms, 729^2 cells p = 4 1.14 / 0.50 ms; operator (projection and
// residual) 64 x 60 x 57 cells p = 4 3.37 / 1.13 ms.
#pragma once

#include <algorithm>
#include <type_traits>

#include "fx.cuh"
#include "internal.h"

namespace dgmg {


// FXM_RESIDUAL_USER: the residual from traces in FP64 (those a caller holds). All other
// kernels exchange traces as they compute them: integers of one exponent per cell, with
// the unused leading bits of each face beside it, so that a reader's sums use all their
// bits (from the exponent alone the errors were three times larger). A face value then
// costs a shift or two on its way in and next to nothing on its way out; converted to FP64
// and back it cost some 40 instructions, a sixth of the smoothing step's: 32^3 cells p = 3
// 98 -> 93 us a step, 23^3 p = 2 V-cycle 149 -> 141 us, 729^2 p = 4 508 -> 501 us.
enum { FXM_SMOOTH = 0, FXM_SMOOTH_FULL = 1, FXM_RESIDUAL = 2, FXM_RESIDUAL_USER = 3 };

template <int DIM, int Q, int SP = 1>
struct FxGeo {
    static constexpr int N = DIM == 3 ? Q * Q : Q;        // nodes of a slab
    static constexpr int NP = N / Q;                      // pencils per lane, face values per lane
    static constexpr int NL = N * Q, NF = N;              // nodes of a cell, of a face
    static constexpr int NFACE = 2 * DIM, FS = 2 * NF, TR = NFACE * FS, NC = 1 << DIM;
    static constexpr int CW = 32 / (Q * SP);              // cells per warp
    static constexpr bool ALL = CW * Q * SP == 32;        // every lane serves a cell
    static constexpr int NW = 4;                          // warps per CTA
    static constexpr int CPB = CW * NW;                   // cells per CTA
    static constexpr int MINB = (Q <= 4 ? 16 : (Q == 5 ? 12 : 8)) / NW;   // CTAs per SM the registers are cut for
    // shared memory, in 8-byte words: slab rows of S, cells of C (strides chosen
    // against bank conflicts of the passes along the first and the last axis)
    static constexpr int S = DIM == 3 ? (N % 2 ? N : N + 2) : (Q | 1);
    static constexpr int C = DIM == 3 && Q % 2 == 0 ? Q * S + 1 : Q * S;
    static constexpr int FDS = Q * Q + Q;                 // factor words per axis (global)
    static constexpr int LW = NFACE * 2 * Q;              // lifting coefficients per cell
    static constexpr int DW = DIM * Q * Q;                // 1D blocks D_a per cell
    // per cell: first the lifting coefficients (and the blocks D_a), then the factors
    __host__ __device__ static constexpr int small_words(int mode) {
        return ((mode == FXM_SMOOTH ? (LW > DIM * FDS ? LW : DIM * FDS)
                                    : (LW + DW > DIM * FDS || mode >= FXM_RESIDUAL ? LW + DW : DIM * FDS)) |
                1);
    }
    // per CTA: M, and for the blocks D_a also K, L, R
    __host__ __device__ static constexpr int tab_words(int mode) { return (mode == FXM_SMOOTH ? 1 : 6) * Q * Q; }
    __host__ __device__ static constexpr int warp_words(int mode) {
        return 2 * CW * C + CW * small_words(mode) + CW * NFACE + 32;   // + exponents: coefficients, lanes (2 x 32)
    }
    __host__ __device__ static constexpr size_t bytes(int mode) { return 8 * (size_t)(tab_words(mode) + NW * warp_words(mode)); }
    __host__ __device__ static constexpr int warp_words_project() { return 2 * CW * C + 32; }
    __host__ __device__ static constexpr size_t bytes_project() { return 8 * (size_t)(NW * warp_words_project()); }
};

__device__ __forceinline__ void fx_cp8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void fx_cp_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// The cell tensors of the warp's cells between global memory (contiguous) and the
// slab rows of shared memory (contiguous too for odd q).
template <int DIM, int Q, int SP>
__device__ __forceinline__ int fx_row_place(int g) {
    using G = FxGeo<DIM, Q, SP>;
    if (G::C == G::NL) return g;
    const int c = g / G::NL, r = g - c * G::NL, row = r / G::N;
    return c * G::C + row * G::S + (r - row * G::N);
}
template <int DIM, int Q, int SP>
__device__ __forceinline__ void fx_stage_in(void *dst, const double *__restrict__ src, int count, int lane) {
    using G = FxGeo<DIM, Q, SP>;
    constexpr int ROUNDS = (G::CW * G::NL + 31) / 32;
    if (ROUNDS <= 32 && count == G::CW * G::NL) {
#pragma unroll
        for (int j = 0; j < ROUNDS; ++j) {
            const int g = lane + 32 * j;
            if (G::CW * G::NL % 32 == 0 || j < ROUNDS - 1 || g < G::CW * G::NL)
                fx_cp8(reinterpret_cast<double *>(dst) + fx_row_place<DIM, Q, SP>(g), src + g);
        }
    } else {
#pragma unroll 4
        for (int g = lane; g < count; g += 32) fx_cp8(reinterpret_cast<double *>(dst) + fx_row_place<DIM, Q, SP>(g), src + g);
    }
}
template <int DIM, int Q, int SP>
__device__ __forceinline__ void fx_store_out(double *__restrict__ dst, const double *src, int count, int lane) {
#pragma unroll 8
    for (int g = lane; g < count; g += 32) dst[g] = src[fx_row_place<DIM, Q, SP>(g)];
}

// The lane's place: cell slot c of the warp, slab k. Lanes beyond CW * q follow slot
// 0 without writing (live = false).
struct FxLane {
    int lane, c, k;
    int sub;                             // which of the SP lanes of its slab
    bool live;
    int *ex;                             // the warp's two rows of lane exponents [2][32]
    int row;                             // the row of the next exchange of them
};
template <int DIM, int Q, int SP>
__device__ __forceinline__ FxLane fx_lane(int *ex) {
    FxLane L;
    L.lane = threadIdx.x & 31;
    L.c = L.lane / (Q * SP);
    L.sub = SP == 1 ? 0 : (L.lane - L.c * (Q * SP)) / Q;
    L.k = L.lane - (L.c * SP + L.sub) * Q;
    L.live = L.c < FxGeo<DIM, Q, SP>::CW;
    if (!L.live) L.c = L.k = L.sub = 0;
    L.ex = ex;
    L.row = 0;
    return L;
}
// The largest v of the cell's lanes; a warp barrier on the way: what the lanes wrote
// to shared memory before is visible after. Calls alternate between two rows, so a
// row is written again only after the barrier of the call in between.
template <int Q>
__device__ __forceinline__ int fx_cell_max(int v, FxLane &L) {
    int *row = L.ex + L.row;
    L.row ^= 32;
    if (L.live) row[L.lane] = v;
    __syncwarp();
    int m = row[L.c * Q];
#pragma unroll
    for (int s = 1; s < Q; ++s) m = imax(m, row[L.c * Q + s]);
    return m;
}

// The same with the smallest of each of four bytes.
template <int Q>
__device__ __forceinline__ unsigned fx_cell_min4(unsigned v, FxLane &L) {
    int *row = L.ex + L.row;
    L.row ^= 32;
    if (L.live) row[L.lane] = (int)v;
    __syncwarp();
    unsigned m = (unsigned)row[L.c * Q];
#pragma unroll
    for (int s = 1; s < Q; ++s) m = __vminu4(m, (unsigned)row[L.c * Q + s]);
    return m;
}

// Pencils of axis a: lane k's pencil p starts at first + p * next and steps by step.
struct FxAxis {
    int first, next, step;
};
template <int DIM, int Q, int SP>
__device__ __forceinline__ FxAxis fx_axis(int a, int k) {
    using G = FxGeo<DIM, Q, SP>;
    FxAxis x;
    const bool last = a == DIM - 1;
    x.first = last ? (DIM == 3 ? Q * k : k) : G::S * k;
    x.next = !last && a == 0 ? Q : 1;
    x.step = last ? G::S : (a == 0 ? 1 : Q);
    return x;
}

// A block in shared memory: value = t 2^e, to be shifted left by n when read (n from
// the largest magnitude of the cell, so that all 60 bits are used). n is negative
// only for the sum of the facet terms, which may exceed 60 bits.
struct FxBlock {
    int e, n;
};
// Largest magnitude of a lane's values, by their high words.
struct FxMag {
    int mx = 0, mn = 0;
    __device__ __forceinline__ void add(long long t) {
        const int h = (int)(t >> 32);
        mx = imax(mx, h);
        mn = imin(mn, h);
    }
    __device__ __forceinline__ int top() const { return imax(mx, ~mn); }
};
__device__ __forceinline__ int fx_headroom(int mag) { return __clz(mag) - 4; }
__device__ __forceinline__ Limb fx_read(long long t, int n) { return limb_of(t << (n & 63)); }
// after a pass whose lanes saw magnitudes mag and whose results have unit e
template <int Q>
__device__ __forceinline__ FxBlock fx_block(const FxMag &mag, int e, FxLane &L) {
    FxBlock b;
    b.n = fx_headroom(fx_cell_max<Q>(mag.top(), L));
    b.e = e;
    return b;
}

// t <- A t along axis a. A[i][m] = src[i * si + m * sm] (limbs of unit ea). Axis and
// matrix are run-time values, so that one copy of the code serves every pass.
template <int DIM, int Q, int SP>
__device__ __forceinline__ FxBlock fx_pass(long long *xc, FxBlock b, int a, const Limb *src, int si, int sm, int ea,
                                           FxLane &L) {
    using G = FxGeo<DIM, Q, SP>;
    const FxAxis ax = fx_axis<DIM, Q, SP>(a, L.k);
    Limb A[Q * Q];
#pragma unroll
    for (int i = 0; i < Q; ++i)
#pragma unroll
        for (int m = 0; m < Q; ++m) A[i * Q + m] = src[i * si + m * sm];
    FxMag mag;
#pragma unroll 1
    for (int p = L.sub; p < G::NP; p += SP) {
        long long *t = xc + ax.first + p * ax.next;
        Acc s[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) acc_zero(s[i]);
#pragma unroll
        for (int m = 0; m < Q; ++m) {
            const Limb x = fx_read(t[m * ax.step], b.n);
#pragma unroll
            for (int i = 0; i < Q; ++i) mac(s[i], A[i * Q + m], x);
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const long long v = acc_value(s[i]);
            if (G::ALL || L.live) t[i * ax.step] = v;
            mag.add(v);
        }
    }
    return fx_block<Q * SP>(mag, b.e - b.n + ea + 64, L);
}

// t <- M t along axis a, M the 1D mass, which is symmetric about its centre: with
// e = x_j + x_j', o = x_j - x_j' (j' = q - 1 - j) the outputs i and i' are
// (E e)_i +- (O o)_i, E = (M_ij + M_ij') / 2, O = (M_ij - M_ij') / 2: half the
// multiply-adds (q = 4: 8 of 16 a pencil), for 2 q additions. GL: the mass is diagonal.
// T: E and O, row-major, or M (GL). |e|, |o| < 2^61 and the h of a row of E and O sum to
// half of M's, so the sums keep the bounds of Acc. With full matrices: residual 243^2
// cells p = 6 GL 120 us (now 110), operator 64^3 p = 4 1192 (1141), smoothing 32^3 p = 3
// 100 (98) a step.
template <int DIM, int Q, int SP>
__device__ __forceinline__ FxBlock fx_mass(long long *xc, FxBlock b, int a, const Limb *T, int eM, bool gl, FxLane &L) {
    using G = FxGeo<DIM, Q, SP>;
    constexpr int H = Q / 2, HE = Q - H;                  // sizes of O and E
    const FxAxis ax = fx_axis<DIM, Q, SP>(a, L.k);
    FxMag mag;
    if (gl) {
#pragma unroll 1
        for (int p = L.sub; p < G::NP; p += SP) {
            long long *t = xc + ax.first + p * ax.next;
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                Acc s;
                acc_zero(s);
                mac(s, T[i * Q + i], fx_read(t[i * ax.step], b.n));
                const long long v = acc_value(s);
                if (G::ALL || L.live) t[i * ax.step] = v;
                mag.add(v);
            }
        }
        return fx_block<Q * SP>(mag, b.e - b.n + eM + 64, L);
    }
    Limb E[HE * HE], O[H * H];
#pragma unroll
    for (int i = 0; i < HE * HE; ++i) E[i] = T[i];
#pragma unroll
    for (int i = 0; i < H * H; ++i) O[i] = T[HE * HE + i];
#pragma unroll 1
    for (int p = L.sub; p < G::NP; p += SP) {
        long long *t = xc + ax.first + p * ax.next;
        Acc se[HE], so[H];
#pragma unroll
        for (int i = 0; i < HE; ++i) acc_zero(se[i]);
#pragma unroll
        for (int i = 0; i < H; ++i) acc_zero(so[i]);
#pragma unroll
        for (int j = 0; j < H; ++j) {
            const long long x = t[j * ax.step] << b.n, y = t[(Q - 1 - j) * ax.step] << b.n;
            const Limb e = limb_of(x + y), o = limb_of(x - y);
#pragma unroll
            for (int i = 0; i < HE; ++i) mac(se[i], E[i * HE + j], e);
#pragma unroll
            for (int i = 0; i < H; ++i) mac(so[i], O[i * H + j], o);
        }
        if constexpr (Q % 2 != 0) {
            const Limb x = fx_read(t[H * ax.step], b.n);
#pragma unroll
            for (int i = 0; i < HE; ++i) mac(se[i], E[i * HE + H], x);
        }
#pragma unroll
        for (int i = 0; i < HE; ++i) {
            const long long ve = acc_value(se[i]);
            if (i < H) {
                const long long vo = acc_value(so[i < H ? i : 0]), v = ve + vo, w = ve - vo;
                if (G::ALL || L.live) {
                    t[i * ax.step] = v;
                    t[(Q - 1 - i) * ax.step] = w;
                }
                mag.add(v);
                mag.add(w);
            } else {
                if (G::ALL || L.live) t[i * ax.step] = ve;
                mag.add(ve);
            }
        }
    }
    return fx_block<Q * SP>(mag, b.e - b.n + eM + 64, L);
}

// Largest biased exponent of the lane's slab of FP64 values.
template <int DIM, int Q, int SP>
__device__ __forceinline__ int fx_slab_top(const double *y, int sub) {
    int mx = 0;
#pragma unroll 4
    for (int i = sub; i < FxGeo<DIM, Q, SP>::N; i += SP) mx = imax(mx, fx_abs_hi(y[i]));
    return mx >> 20;
}

// Unit of the block of the cell's FP64 values y (in the lanes' slabs), from the largest
// biased exponent of this lane's values; a warp barrier. A cell that looks like zeros may
// hold subnormal values: their own largest bit decides then.
template <int DIM, int Q, int SP>
__device__ __forceinline__ int fx_cell_unit(int mine, const double *y, FxLane &L) {
    const int top = fx_cell_max<Q * SP>(mine, L);
    int unit = fx_unit(top);
    if (__any_sync(0xffffffffu, top == 0)) {
        int bits = 0;                                    // of the largest subnormal value
#pragma unroll 1
        for (int i = L.sub; i < FxGeo<DIM, Q, SP>::N; i += SP) {
            const int h = fx_abs_hi(y[i]), l = lo_word(y[i]);
            bits = imax(bits, h != 0 ? 64 - clz32(h) : 32 - clz32(l));
        }
        bits = fx_cell_max<Q * SP>(bits, L);
        if (top == 0 && bits > 0) unit = 1 - FX_UNIT - (53 - bits);
    }
    return unit;
}

// f(std::true_type) where the blocks of all the warp's cells hold normal numbers only, by
// their exponent e, else f(std::false_type).
template <typename F>
__device__ __forceinline__ void fx_by_range(int e, F f) {
    if (__any_sync(0xffffffffu, !fx_safe(e)))
        f(std::false_type{});
    else
        f(std::true_type{});
}

// The lane's slab of FP64 values as block values of that unit.
template <int DIM, int Q, int SP>
__device__ __forceinline__ void fx_to_block(long long *xs, const double *ys, int unit, const FxLane &L) {
    constexpr int N = FxGeo<DIM, Q, SP>::N;
    const int ev = unit + FX_UNIT;
    if (__any_sync(0xffffffffu, ev < FX_LOW)) {
#pragma unroll 1
        for (int i = L.sub; i < N; i += SP) {
            const long long v = fx_from_any(ys[i], ev);
            if (L.live) xs[i] = v;
        }
        return;
    }
#pragma unroll 4
    for (int i = L.sub; i < N; i += SP) {
        const long long v = fx_from(ys[i], ev);
        if (L.live) xs[i] = v;
    }
}

// Per cell after the traces {e, h[axis]}: values count 2^e (GL: 2^(e + eV + 64)),
// derivatives along axis a 2^(e + eT[a] + 64); h packs the unused leading bits (of 60) of
// the axis' traces, byte 2 side + (0 value, 1 derivative).
template <int DIM, int Q, int SP, typename P>
__device__ __forceinline__ auto fx_trace_units(P *tr, int64_t ncell) {
    using I = typename std::conditional<std::is_const<P>::value, const int4, int4>::type;
    return reinterpret_cast<I *>(tr + ncell * FxGeo<DIM, Q, SP>::TR);
}
constexpr int FX_NO_TRACE = FX_NONE / 2;     // exponents below: all values are 0

// Traces of the cell from its block in shared memory: per axis and side, value and
// +axis derivative; derivatives by dot products, values the end nodes (GLL) or dot
// products (GL). USER: as FP64, the end nodes' values from the cell's FP64 values yc.
template <int DIM, int Q, int SP, bool USER = false>
__device__ __forceinline__ void fx_all_traces(const FxTab &tab, const FxConst &cst, const long long *xc, FxBlock b,
                                              FxLane &L, bool write, int64_t cell, double *__restrict__ tr,
                                              const double *yc = nullptr) {
    using G = FxGeo<DIM, Q, SP>;
    const int e = b.e - b.n;
    double *cell_tr = tr + cell * G::TR;
    unsigned room[3] = {0, 0, 0};
#pragma unroll 1
    for (int a = 0; a < DIM; ++a) {
        const FxAxis ax = fx_axis<DIM, Q, SP>(a, L.k);
        Limb d[2][Q];
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int i = 0; i < Q; ++i) d[s][i] = cst.dt[a][s][i];
        const int ed = e + cst.eT[a] + 64;
        double *out = cell_tr + 2 * a * G::FS + L.k * G::NP;
        FxMag mag[2][2];
        auto put_at = [&](int s, int c, int p, long long w, int ew) {
            double *to = out + s * G::FS + c * G::NF + p;
            if (!USER) mag[s][c].add(w);
            if (!write) return;
            if (USER)
                *to = fx_to(w, ew);
            else
                *reinterpret_cast<long long *>(to) = w;
        };
#pragma unroll 1
        for (int p = L.sub; p < G::NP; p += SP) {
            const long long *t = xc + ax.first + p * ax.next;
            auto put = [&](int s, int c, long long w, int ew) { put_at(s, c, p, w, ew); };
            Limb x[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) x[i] = fx_read(t[i * ax.step], b.n);
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                Acc v;
                acc_zero(v);
#pragma unroll
                for (int i = 0; i < Q; ++i) mac(v, d[s][i], x[i]);
                put(s, 1, acc_value(v), ed);
                if (tab.gl) {
                    acc_zero(v);
#pragma unroll
                    for (int i = 0; i < Q; ++i) mac(v, tab.v[s][i], x[i]);
                    put(s, 0, acc_value(v), e + tab.eV + 64);
                } else if (USER) {
                    if (write) out[s * G::FS + p] = yc[(t - xc) + (s ? Q - 1 : 0) * ax.step];
                } else {
                    put(s, 0, t[(s ? Q - 1 : 0) * ax.step] << b.n, e);
                }
            }
        }
        if (!USER) {
            unsigned w = 0;
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int c = 0; c < 2; ++c) w |= (unsigned)imax(fx_headroom(mag[s][c].top()), 0) << (16 * s + 8 * c);
            w = fx_cell_min4<Q * SP>(w, L);
            room[0] = a == 0 ? w : room[0];
            room[1] = a == 1 ? w : room[1];
            room[2] = a == 2 ? w : room[2];
        }
    }
    if (!USER && write && L.k == 0)
        fx_trace_units<DIM, Q, SP>(tr, cst.ncell)[cell] = make_int4(e, (int)room[0], (int)room[1], (int)room[2]);
}

__device__ __forceinline__ void load_batch_desc(const BatchDG<double> *__restrict__ src, BatchDG<double> *dst) {
    static_assert(sizeof(BatchDG<double>) % 8 == 0, "descriptor copied in 8-byte words");
    const unsigned long long *s = reinterpret_cast<const unsigned long long *>(src);
    unsigned long long *d = reinterpret_cast<unsigned long long *>(dst);
    for (int i = threadIdx.x; i < (int)(sizeof(BatchDG<double>) / 8); i += blockDim.x) d[i] = s[i];
    __syncthreads();
}

template <int DIM>
__device__ __forceinline__ void fx_cell_coords(int64_t cell, const int *n, int *ci) {
    if (cell <= 0x7fffffff) {
        const unsigned u = (unsigned)cell, r = u / (unsigned)n[0];
        ci[0] = (int)(u - r * (unsigned)n[0]);
        ci[1] = DIM == 3 ? (int)(r % (unsigned)n[1]) : (int)r;
        ci[2] = DIM == 3 ? (int)(r / (unsigned)n[1]) : 0;
        return;
    }
    ci[0] = (int)(cell % n[0]);
    const int64_t r = cell / n[0];
    ci[1] = DIM == 3 ? (int)(r % n[1]) : (int)r;
    ci[2] = DIM == 3 ? (int)(r / n[1]) : 0;
}

// Smoothing step (FXM_SMOOTH: exact blocks, FXM_SMOOTH_FULL: the block of an
// interior cell, so the whole residual is formed first) or residual of the warp's
// cells [cell0, cell0 + CW) of the level.
//
// Exact blocks: A u = A_KK u + N u_nb, so u <- (1 - w) u + w A_KK^-1 (b - N u_nb);
// A_KK^-1 by fast diagonalisation (Kt_a S_a = M_a S_a Lambda_a): S^T along every
// axis, times the table omega / (sum of eigenvalues), S along every axis. fd: the
// cell's limbs of S per axis, their exponents in the words after them (axis 0 also
// the table's); linv: the table.
// flags: SM_ZERO: the iterate is 0 (u and its traces are not read); SM_NO_TRACES:
// the new traces are not written. mode (residual): RES_*.
template <int DIM, int Q, int SP, int MODE>
__device__ __forceinline__ void fx_cells_body(const FxTab &tab, const FxConst &cst, const Limb *sTab, long long *smem,
                                              int64_t cell0, int flags, int mode, double *__restrict__ u,
                                              const double *__restrict__ b, const double *__restrict__ kappa,
                                              const double *__restrict__ fd, const double *__restrict__ linv,
                                              const double *__restrict__ tr_in, double *__restrict__ tr_out,
                                              double *__restrict__ r, double *__restrict__ corners) {
    using G = FxGeo<DIM, Q, SP>;
    constexpr int N = G::N, NP = G::NP, NL = G::NL, NFACE = G::NFACE, SW = G::small_words(MODE);
    constexpr bool SMOOTH = MODE < FXM_RESIDUAL, FULL = MODE != FXM_SMOOTH, USER = MODE == FXM_RESIDUAL_USER;
    long long *X = smem;                                  // the block the passes work on
    long long *Y = X + G::CW * G::C;                      // u or b on their way in, the result on its way out
    Limb *small = reinterpret_cast<Limb *>(Y + G::CW * G::C);   // coefficients and D_a, later the factors
    int *sLE = reinterpret_cast<int *>(small + G::CW * SW);     // coefficient exponents [cell][face][field]
    FxLane L = fx_lane<DIM, Q, SP>(sLE + G::CW * NFACE * 2);
    const int ncl = (int)(cst.ncell - cell0 < G::CW ? cst.ncell - cell0 : G::CW);
    const bool active = L.live && L.c < ncl;
    const int64_t cell = cell0 + (L.c < ncl ? L.c : 0);
    const bool zero = SMOOTH && (flags & SM_ZERO) != 0;
    const bool has_b = SMOOTH || (mode & RES_HAS_B) != 0;
    long long *xc = X + L.c * G::C;
    double *yc = reinterpret_cast<double *>(Y + L.c * G::C), *ys = yc + L.k * G::S;   // the cell, the lane's slab
    long long *xs = xc + L.k * G::S;
    Limb *mine = small + L.c * SW;

    // in flight from the start: u where the residual of the iterate needs it, else b
    fx_stage_in<DIM, Q, SP>(Y, (FULL && !zero ? u : b) + cell0 * NL, FULL && !zero ? ncl * NL : (has_b ? ncl * NL : 0),
                        L.lane);
    auto stage_factors = [&]() {
        if constexpr (SMOOTH) {
            constexpr int W = DIM * G::FDS;
#pragma unroll 4
            for (int g = L.lane; g < ncl * W; g += 32) {
                const int c = g / W;
                fx_cp8(small + c * SW + (g - c * W), fd + cell0 * W + g);
            }
        }
    };

    FxBlock t{FX_NONE, 0};
    if (zero) {
        stage_factors();
    } else {
        int ci[3];
        fx_cell_coords<DIM>(cell, cst.n, ci);
        const double *kf = cst.kfac + cell * NFACE;
        // bit f: face f has a neighbour; its traces for this lane's pencils
        int mask = 0;
#pragma unroll
        for (int a = 0; a < DIM; ++a) mask |= (ci[a] > 0 ? 1 << (2 * a) : 0) | (ci[a] < cst.n[a] - 1 ? 2 << (2 * a) : 0);
        const int64_t s1 = cst.n[0], s2 = s1 * cst.n[1];
        // (a boundary face: the cell's own, read and not used)
        auto face = [&](int a, int s, bool in) {
            const int64_t st = a == 0 ? 1 : (a == 1 ? s1 : s2);
            return tr_in + (in ? cell + (s ? st : -st) : cell) * G::TR + (2 * a + (s ^ 1)) * G::FS + L.k * NP;
        };
        // lifting coefficients: facet coefficient x vector, node k of every vector by
        // lane k; the unit of the facet terms from the largest product of a
        // coefficient's and a trace's exponent
        // units of the neighbour's value and derivative traces (USER: from the high words
        // of the lane's values, requested at once for every face)
        int ug[NFACE], uh[NFACE], rg[NFACE], rh[NFACE];   // units, and unused leading bits
#pragma unroll
        for (int f = 0; f < NFACE; ++f) {
            const int a = f >> 1;
            if constexpr (USER) {
                const double *nb = face(a, f & 1, ((mask >> f) & 1) != 0);
                int mg = 0, mh = 0;
                bool sg = false, sh = false;              // some value is not 0 (it may be subnormal)
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const double g = __ldg(nb + p), h = __ldg(nb + G::NF + p);
                    mg = imax(mg, fx_abs_hi(g));
                    mh = imax(mh, fx_abs_hi(h));
                    sg = sg || fx_some(g);
                    sh = sh || fx_some(h);
                }
                ug[f] = fx_unit(imax(mg >> 20, sg ? 1 : 0));
                uh[f] = fx_unit(imax(mh >> 20, sh ? 1 : 0));
                rg[f] = rh[f] = 0;
            } else {
                const int64_t st = a == 0 ? 1 : (a == 1 ? s1 : s2);
                const int64_t nb = (mask >> f) & 1 ? cell + (f & 1 ? st : -st) : cell;
                const int4 en = __ldg(fx_trace_units<DIM, Q, SP>(tr_in, cst.ncell) + nb);
                const unsigned w = (unsigned)(a == 0 ? en.y : (a == 1 ? en.z : en.w)) >> (f & 1 ? 0 : 16);
                ug[f] = en.x + (tab.gl ? tab.eV + 64 : 0);
                uh[f] = en.x + cst.eT[a] + 64;
                rg[f] = (int)(w & 255u);
                rh[f] = (int)(w >> 8 & 255u);
            }
        }
        int top = FX_NONE;
#pragma unroll
        for (int f = 0; f < NFACE; ++f) {
            const int a = f >> 1, s = f & 1;
            const bool in = (mask >> f) & 1;
            const double v = in ? kf[f] : 0.0;
            const int ev = fx_abs_hi(v) >> 20;
            const Limb x = limb_of(fx_from(v, ev));
            Acc g, h;
            acc_zero(g);
            acc_zero(h);
            mac(g, tab.cG[s][L.k], x);
            mac(h, cst.cH[a][s][L.k], x);
            // |acc_value| < 2^57: shifted by 4 the h of a coefficient is below 2^29
            const int lg = fx_unit(ev) + tab.eG + 64 - 4, lh = fx_unit(ev) + cst.eH[a] + 64 - 4;
            if (L.live) {
                mine[(f * 2 + 0) * Q + L.k] = limb_of(acc_value(g) << 4);
                mine[(f * 2 + 1) * Q + L.k] = limb_of(acc_value(h) << 4);
                if (L.k == 0) {                          // the unit of a product, or (USER) of the coefficients
                    sLE[(L.c * NFACE + f) * 2 + 0] = USER ? lg : lg + ug[f];
                    sLE[(L.c * NFACE + f) * 2 + 1] = USER ? lh : lh + uh[f];
                }
            }
            if (in && ug[f] > FX_NO_TRACE) top = imax(top, ug[f] - rg[f] + lg + 64);
            if (in && uh[f] > FX_NO_TRACE) top = imax(top, uh[f] - rh[f] + lh + 64);
        }
        int ed = FX_NONE;
        if constexpr (FULL) {
            // the cell's 1D blocks D_a = alpha K + beta_L L + beta_R R, row k by lane k
            const double kK = __ldg(kappa + cell);
            int mx = 0;
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                mx = imax(mx, fx_abs_hi(cst.sa[a] * kK));
#pragma unroll
                for (int s = 0; s < 2; ++s) mx = imax(mx, fx_abs_hi(kf[2 * a + s]));
            }
            const int ev = mx >> 20;
            const Limb *rows = sTab + Q * Q + L.k * Q;
#pragma unroll 1
            for (int a = 0; a < DIM; ++a) {
                const double al = cst.sa[a] * kK;
                const bool in0 = (mask >> (2 * a)) & 1, in1 = (mask >> (2 * a + 1)) & 1;
                const Limb x = limb_of(fx_from(al, ev)), y = limb_of(fx_from(in0 ? kf[2 * a] : al, ev)),
                           z = limb_of(fx_from(in1 ? kf[2 * a + 1] : al, ev));
                const Limb *rowL = rows + (in0 ? 1 : 2) * Q * Q, *rowR = rows + (in1 ? 3 : 4) * Q * Q;
#pragma unroll
                for (int m = 0; m < Q; ++m) {
                    Acc s;
                    acc_zero(s);
                    mac(s, rows[m], x);
                    mac(s, rowL[m], y);
                    mac(s, rowR[m], z);
                    // row sums of |acc_value| stay below 2^58: shifted by 4, the h of a row sum to 2^30
                    if (L.live) mine[G::LW + (a * Q + L.k) * Q + m] = limb_of(acc_value(s) << 4);
                }
            }
            ed = fx_unit(ev) + tab.eD + 64 - 4;
            fx_cp_wait();
            __syncwarp();
        }
        // one unit E for the whole sum: |D u| < 2^58 and the facet terms < 2^59 per axis,
        // so the sum over the axes stays below 2^62
        int E = fx_cell_max<Q * SP>(top, L);
        if constexpr (FULL) {
            E = imax(E, fx_cell_unit<DIM, Q, SP>(fx_slab_top<DIM, Q, SP>(ys, L.sub), ys, L) + ed + 64);
            // u as integers of the unit that makes D u come out in E
            fx_to_block<DIM, Q, SP>(reinterpret_cast<long long *>(ys), ys, E - ed - 64, L);
            __syncwarp();
        }
        FxMag mag;
#pragma unroll 1
        for (int a = 0; a < DIM; ++a) {
            const FxAxis ax = fx_axis<DIM, Q, SP>(a, L.k);
            if (a == DIM - 1 || (SP > 1 && a > 0)) __syncwarp();   // this axis crosses the lanes' parts
            mag = FxMag();
            Limb B[FULL ? Q * Q : 1], cf[2][2][Q];
            if constexpr (FULL) {
#pragma unroll
                for (int i = 0; i < Q * Q; ++i) B[i] = mine[G::LW + a * Q * Q + i];
            }
            int ev[2][2];
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    // the exponent the trace is converted with, or the places it is shifted to the right
                    ev[s][c] = E - 64 - sLE[(L.c * NFACE + 2 * a + s) * 2 + c];
                    ev[s][c] = USER ? ev[s][c] + FX_UNIT : imin(imax(ev[s][c], -60), 63);
#pragma unroll
                    for (int i = 0; i < Q; ++i) cf[s][c][i] = mine[((2 * a + s) * 2 + c) * Q + i];
                }
            const bool in[2] = {((mask >> (2 * a)) & 1) != 0, ((mask >> (2 * a + 1)) & 1) != 0};
            const double *nb[2] = {face(a, 0, in[0]), face(a, 1, in[1])};
#pragma unroll 1
            for (int p = L.sub; p < NP; p += SP) {
                long long *o = xc + ax.first + p * ax.next;
                const long long *y = Y + L.c * G::C + ax.first + p * ax.next;
                Limb g[2][2];
#pragma unroll
                for (int s = 0; s < 2; ++s)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const double w = __ldg(nb[s] + c * G::NF + p);
                        const long long v = USER ? fx_from_any(w, ev[s][c])
                                                 : (__double_as_longlong(w) << imax(-ev[s][c], 0)) >> imax(ev[s][c], 0);
                        g[s][c] = limb_of(in[s] ? v : 0ll);
                    }
                Acc v[Q];
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    acc_zero(v[i]);
                    if (a > 0) v[i].hh = o[i * ax.step];
#pragma unroll
                    for (int s = 0; s < 2; ++s)
#pragma unroll
                        for (int c = 0; c < 2; ++c) mac(v[i], cf[s][c][i], g[s][c]);
                }
                if constexpr (FULL) {                    // a sum of its own: m has room for q terms
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        v[i].hh = acc_value(v[i]);
                        v[i].m = 1ll << 31;
                    }
#pragma unroll
                    for (int m = 0; m < Q; ++m) {
                        const Limb x = limb_of(y[m * ax.step]);
#pragma unroll
                        for (int i = 0; i < Q; ++i) mac(v[i], B[i * Q + m], x);
                    }
                }
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const long long w = acc_value(v[i]);
                    if (G::ALL || L.live) o[i * ax.step] = w;
                    mag.add(w);
                }
            }
        }
        t = fx_block<Q * SP>(mag, E, L);
        // more than 60 bits somewhere (the bound on the sum is 2^62): shift those cells
        if (__any_sync(0xffffffffu, t.n < 0)) {
            const int d = imax(-t.n, 0);
#pragma unroll 4
            for (int i = L.sub; i < N; i += SP)
                if (G::ALL || L.live) xs[i] >>= d;
            t.e += d;
            t.n = imax(t.n, 0);
            __syncwarp();
        }
        // the coefficients are used: the factors (or b) while M is applied
        stage_factors();
        if (FULL && has_b) fx_stage_in<DIM, Q, SP>(Y, b + cell0 * NL, ncl * NL, L.lane);
    }
    // M along every axis; t <- b - t; S^T along every axis; the table; S along every axis
    const Limb *myF = mine;
    // The residual on its way out keeps the bits of b: a subtraction in FP64 per node. (As
    // a block it has those of the cell's largest value, so that u = 0 did not give b back.)
    const bool write_r = !SMOOTH && has_b && (mode & RES_WRITE_R) != 0;
    auto difference = [&](double bi, double w) { return mode & RES_NEGATE ? w - bi : bi - w; };
    auto subtract_from_b = [&]() {                        // t = A u (or its neighbours' part); in the lane's slab
        fx_cp_wait();
        __syncwarp();
        const int tb = fx_cell_unit<DIM, Q, SP>(fx_slab_top<DIM, Q, SP>(ys, L.sub), ys, L);
        const int te = t.e - t.n, E = imax(tb, te) + 1;
        const int ev = E + FX_UNIT;
        FxMag mag;
        auto at = [&](int i, long long v) {               // v: b as a block value
            const long long ti = xs[i];
            if (!zero) v -= fx_shr(ti << t.n, E - te);
            if (G::ALL || L.live) xs[i] = v;
            mag.add(v);
        };
        if (__any_sync(0xffffffffu, ev < FX_LOW)) {
#pragma unroll 1
            for (int i = L.sub; i < N; i += SP) at(i, fx_from_any(ys[i], ev));
        } else {
#pragma unroll 4
            for (int i = L.sub; i < N; i += SP) at(i, fx_from(ys[i], ev));
        }
        t = fx_block<Q * SP>(mag, E, L);
    };
#pragma unroll 1
    for (int k = zero ? DIM : 0; k < (SMOOTH ? 3 * DIM : DIM); ++k) {
        if (SMOOTH && k == DIM) {
            subtract_from_b();
            // the table into Y (every lane has read b)
            fx_stage_in<DIM, Q, SP>(Y, linv + cell0 * NL, ncl * NL, L.lane);
        }
        if (SMOOTH && k == 2 * DIM) {
            fx_cp_wait();
            __syncwarp();
            const long long *li = reinterpret_cast<const long long *>(ys);
            int least = FX_SCALED_MOST;
#pragma unroll 4
            for (int i = L.sub; i < N; i += SP) least = imin(least, fx_scaled_below(xs[i], li[i]));
            least = FX_SCALED_MOST - fx_cell_max<Q * SP>(FX_SCALED_MOST - least, L);
#pragma unroll 4
            for (int i = L.sub; i < N; i += SP) {
                const long long v = fx_scaled(xs[i], li[i], least);
                if (G::ALL || L.live) xs[i] = v;
            }
            t = FxBlock{t.e + myF[Q * Q + 1].h - least, 2};   // (the largest is between 2^56 and 2^58)
            __syncwarp();
            // the previous iterate into Y (every lane has read the table)
            if (!zero) fx_stage_in<DIM, Q, SP>(Y, u + cell0 * NL, ncl * NL, L.lane);
        }
        const int a = k < DIM ? DIM - 1 - k : (k < 2 * DIM ? k - DIM : 3 * DIM - 1 - k);
        if (k < DIM) {
            t = fx_mass<DIM, Q, SP>(xc, t, a, sTab, tab.eM, tab.gl != 0, L);
        } else if constexpr (SMOOTH) {
            const bool trans = k < 2 * DIM;
            const Limb *src = myF + a * G::FDS;
            t = fx_pass<DIM, Q, SP>(xc, t, a, src, trans ? 1 : Q, trans ? Q : 1, src[Q * Q].h, L);
        }
    }
    if (!SMOOTH && has_b) {
        if (mode & RES_CORNERS) {
            if (write_r) {                               // (both are wanted by callers' calls only)
                fx_cp_wait();
                __syncwarp();
#pragma unroll 1
                for (int i = L.sub; i < N; i += SP)
                    if (active) r[cell * NL + L.k * N + i] = difference(ys[i], fx_to(xs[i], t.e));
            }
            subtract_from_b();
        } else {
            fx_cp_wait();
            __syncwarp();
            fx_by_range(t.e, [&](auto safe) {
#pragma unroll 4
                for (int i = L.sub; i < N; i += SP) {
                    const double v = difference(ys[i], fx_to<decltype(safe)::value>(xs[i], t.e));
                    if (L.live) ys[i] = v;
                }
            });
        }
    }
    const bool traces = SMOOTH && !(flags & SM_NO_TRACES);
    bool in_y = write_r;                                  // the result is in Y
    if constexpr (SMOOTH) {
        // the last pass ran along axis 0, in the lane's own slab
        if (!zero) {
            // u <- keep u + t node by node in FP64 (u keeps its bits, whatever its cell's
            // largest value is); the block for the traces is read from the result
            fx_cp_wait();
            __syncwarp();
            int top = 0;
            fx_by_range(t.e, [&](auto safe) {
#pragma unroll 4
                for (int i = L.sub; i < N; i += SP) {
                    const double v = fma(cst.keep, ys[i], fx_to<decltype(safe)::value>(xs[i], t.e));
                    if (L.live) ys[i] = v;
                    top = imax(top, fx_abs_hi(v));
                }
            });
            in_y = true;
            if (traces) {
                t = FxBlock{fx_cell_unit<DIM, Q, SP>(top >> 20, ys, L), 0};
                fx_to_block<DIM, Q, SP>(xs, ys, t.e, L);
            }
        }
    }
    // the result leaves through Y
    if (SMOOTH || ((mode & RES_WRITE_R) && !(write_r && (mode & RES_CORNERS)))) {
        // without b the block is A u: the residual b - A u is its negative
        const bool neg = !SMOOTH && !(mode & RES_NEGATE);
        if (!in_y)
            fx_by_range(t.e, [&](auto safe) {
#pragma unroll 4
                for (int i = L.sub; i < N; i += SP) {
                    const double v = fx_to<decltype(safe)::value>(neg ? -xs[i] : xs[i], t.e);
                    if (L.live) ys[i] = v;
                }
            });
        __syncwarp();
        fx_store_out<DIM, Q, SP>((SMOOTH ? u : r) + cell0 * NL, reinterpret_cast<const double *>(Y), ncl * NL, L.lane);
    }
    if constexpr (SMOOTH) {
        if (traces) fx_all_traces<DIM, Q, SP>(tab, cst, xc, t, L, active, cell, tr_out);
    } else if (mode & RES_CORNERS) {
        // corner sums of b - A u: hat values along the slab's axes, then over the slabs
        constexpr int NS = DIM == 3 ? 4 : 2;             // sums per slab
        long long y[NS], s0[2][NP];
        FxMag mag;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            Limb x[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) x[i] = fx_read(xs[i + Q * j], t.n);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                Acc s;
                acc_zero(s);
#pragma unroll
                for (int i = 0; i < Q; ++i) mac(s, tab.hat[c][i], x[i]);
                s0[c][j] = acc_value(s);
                mag.add(s0[c][j]);
            }
        }
        int e = t.e - t.n + tab.eHat + 64, n = fx_headroom(fx_cell_max<Q * SP>(mag.top(), L));
        if constexpr (DIM == 3) {
            mag = FxMag();
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                Acc s;
                acc_zero(s);
#pragma unroll
                for (int j = 0; j < Q; ++j) mac(s, tab.hat[c >> 1][j], limb_of(s0[c & 1][j] << n));
                y[c] = acc_value(s);
                mag.add(y[c]);
            }
            e += tab.eHat + 64 - n;
            n = fx_headroom(fx_cell_max<Q * SP>(mag.top(), L));
        } else {
            y[0] = s0[0][0];
            y[1] = s0[1][0];
        }
        __syncwarp();
        if (L.live) {
#pragma unroll
            for (int c = 0; c < NS; ++c) xs[c] = y[c];
        }
        __syncwarp();
        if (active) {
            for (int id = L.k; id < G::NC; id += Q) {
                Acc s;
                acc_zero(s);
#pragma unroll
                for (int m = 0; m < Q; ++m)
                    mac(s, tab.hat[id >> (DIM - 1)][m], limb_of(xc[m * G::S + (id & (NS - 1))] << n));
                const long long v = acc_value(s);
                const bool neg = has_b == ((mode & RES_NEGATE) != 0);
                corners[cell * G::NC + id] = fx_to(neg ? -v : v, e - n + tab.eHat + 64);
            }
        }
    }
}

template <int DIM, int Q, int SP, int MODE>
__device__ __forceinline__ const Limb *fx_stage_tables(const FxTab &tab, long long *smem) {
    Limb *s = reinterpret_cast<Limb *>(smem);
    constexpr int H = Q / 2, HE = Q - H;
    for (int i = threadIdx.x; i < Q * Q; i += blockDim.x) {
        // the mass as fx_mass reads it: E, then O (GL: M)
        auto whole = [&](int r, int c) { return ((long long)tab.M[r * Q + c].h << 32) + tab.M[r * Q + c].l; };
        if (tab.gl) {
            s[i] = tab.M[i];
        } else if (i < HE * HE) {
            const int r = i / HE, c = i - r * HE;
            const long long a = whole(r, c), b = whole(r, Q - 1 - c);
            s[i] = limb_of((a & b) + ((a ^ b) >> 1));    // their mean (the middle one twice: its double has 65 bits)
        } else if (i < HE * HE + H * H) {
            const int r = (i - HE * HE) / H, c = i - HE * HE - r * H;
            s[i] = limb_of((whole(r, c) - whole(r, Q - 1 - c)) >> 1);
        }
        if (MODE != FXM_SMOOTH) {
            s[Q * Q + i] = tab.K[i];
            s[2 * Q * Q + i] = tab.L[0][i];
            s[3 * Q * Q + i] = tab.L[1][i];
            s[4 * Q * Q + i] = tab.R[0][i];
            s[5 * Q * Q + i] = tab.R[1][i];
        }
    }
    __syncthreads();
    return s;
}

template <int DIM, int Q, int SP, int MODE>
__global__ void __launch_bounds__(FxGeo<DIM, Q, SP>::NW * 32, FxGeo<DIM, Q, SP>::MINB)
    k_fx_cells(const __grid_constant__ FxTab tab, const __grid_constant__ FxConst cst, int flags, int mode, double *u,
               const double *b, const double *__restrict__ kappa, const double *__restrict__ fd,
               const double *__restrict__ linv, const double *__restrict__ tr_in, double *__restrict__ tr_out, double *r,
               double *__restrict__ corners) {
    using G = FxGeo<DIM, Q, SP>;
    extern __shared__ __align__(16) long long smem_fx[];
    const Limb *sTab = fx_stage_tables<DIM, Q, SP, MODE>(tab, smem_fx);
    const int warp = threadIdx.x >> 5;
    const int64_t cell0 = (int64_t)blockIdx.x * G::CPB + warp * G::CW;
    if (cell0 >= cst.ncell) return;
    fx_cells_body<DIM, Q, SP, MODE>(tab, cst, sTab, smem_fx + G::tab_words(MODE) + warp * G::warp_words(MODE), cell0, flags, mode, u, b,
                                kappa, fd, linv, tr_in, tr_out, r, corners);
}

// Batched form: work item k serves the CPB cells from map[k].cell0 of instance
// map[k].inst. Persistent CTAs stride through the items; the barriers end every
// warp's use of the descriptor and of its staging memory.
template <int DIM, int Q, int SP, int MODE>
__global__ void __launch_bounds__(FxGeo<DIM, Q, SP>::NW * 32, FxGeo<DIM, Q, SP>::MINB)
    k_fx_cells_batch(const __grid_constant__ FxTab tab, const BatchDG<double> *__restrict__ D,
                     const BlockMap *__restrict__ map, int nblocks, int flags, int mode, double *u, const double *b,
                     double *r, int cur) {
    using G = FxGeo<DIM, Q, SP>;
    extern __shared__ __align__(16) long long smem_fx[];
    __shared__ __align__(16) BatchDG<double> sd;
    const Limb *sTab = fx_stage_tables<DIM, Q, SP, MODE>(tab, smem_fx);
    const int warp = threadIdx.x >> 5;
    long long *mine = smem_fx + G::tab_words(MODE) + warp * G::warp_words(MODE);
    for (int k = blockIdx.x; k < nblocks; k += gridDim.x) {
        if (k != (int)blockIdx.x) __syncthreads();
        const BlockMap m = map[k];
        load_batch_desc(D + m.inst, &sd);
        const int64_t cell0 = (int64_t)m.cell0 + warp * G::CW;
        if (cell0 < sd.c.ncell) {
            const int64_t o = sd.off * G::NL;
            fx_cells_body<DIM, Q, SP, MODE>(tab, sd.c, sTab, mine, cell0, flags, mode, u + o, b ? b + o : nullptr, sd.kappa,
                                        sd.fd, sd.linv, sd.tr[cur], sd.tr[cur ^ 1], r ? r + o : nullptr, sd.corners);
        }
    }
}

// Warm-up projection of the warp's cells: optionally u += P e (the multilinear hats
// of the cell's corner values), then the traces.
template <int DIM, int Q, int SP, bool USER = false>
__device__ __forceinline__ void fx_project_body(const FxTab &tab, const FxConst &cst, long long *smem, int64_t cell0,
                                                double *u, const double *__restrict__ e0, double *__restrict__ tr) {
    using G = FxGeo<DIM, Q, SP>;
    constexpr int N = G::N, NP = G::NP, NL = G::NL;
    long long *X = smem, *Y = X + G::CW * G::C;
    FxLane L = fx_lane<DIM, Q, SP>(reinterpret_cast<int *>(Y + G::CW * G::C));
    const int ncl = (int)(cst.ncell - cell0 < G::CW ? cst.ncell - cell0 : G::CW);
    const bool active = L.live && L.c < ncl;
    const int64_t cell = cell0 + (L.c < ncl ? L.c : 0);
    long long *xc = X + L.c * G::C, *xs = xc + L.k * G::S;
    double *ys = reinterpret_cast<double *>(Y + L.c * G::C) + L.k * G::S;
    fx_stage_in<DIM, Q, SP>(Y, u + cell0 * NL, ncl * NL, L.lane);
    double ec[G::NC];
    if (e0) {
        int ci[3];
        fx_cell_coords<DIM>(cell, cst.n, ci);
#pragma unroll
        for (int c = 0; c < G::NC; ++c) {
            bool in = true;
            int64_t id = 0, stride = 1;
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                const int v = ci[a] + ((c >> a) & 1);
                in = in && v >= 1 && v <= cst.n[a] - 1;
                id += (int64_t)(v - 1) * stride;
                stride *= cst.n[a] - 1;
            }
            ec[c] = in ? e0[id] : 0.0;
        }
    }
    fx_cp_wait();
    __syncwarp();
    int top = 0;                                          // of the new u, by its high words
    if (e0) {
        int mx = 0;
        bool some = false;
#pragma unroll
        for (int c = 0; c < G::NC; ++c) {
            mx = imax(mx, fx_abs_hi(ec[c]));
            some = some || fx_some(ec[c]);
        }
        const int ev = imax(mx >> 20, some ? 1 : 0);
        int ee = fx_unit(ev);
        constexpr int NH = G::NC / 2;
        long long z[NH];                                  // corners of the slab: the last axis interpolated at k
        FxMag mag;
#pragma unroll
        for (int c = 0; c < NH; ++c) {
            Acc s;
            acc_zero(s);
            mac(s, tab.hat[0][L.k], limb_of(fx_from_any(ec[c], ev)));
            mac(s, tab.hat[1][L.k], limb_of(fx_from_any(ec[c + NH], ev)));
            z[c] = acc_value(s);
            mag.add(z[c]);
        }
        const int n = fx_headroom(fx_cell_max<Q * SP>(mag.top(), L));
        ee += tab.eHat + 64 - n;
        const int ew = ee + (DIM - 1) * (tab.eHat + 64);
#pragma unroll 1
        for (int p = L.sub; p < NP; p += SP) {
            Limb y[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                if constexpr (DIM == 3) {
                    Acc s;
                    acc_zero(s);
                    mac(s, tab.hat[0][p], limb_of(z[c] << n));
                    mac(s, tab.hat[1][p], limb_of(z[c + 2] << n));
                    y[c] = limb_of(acc_value(s));
                } else {
                    y[c] = limb_of(z[c] << n);
                }
            }
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                Acc s;
                acc_zero(s);
                mac(s, tab.hat[0][i], y[0]);
                mac(s, tab.hat[1][i], y[1]);
                // node by node in FP64: u keeps its bits, whatever its cell's largest value is
                const double v = ys[i + Q * p] + fx_to(acc_value(s), ew);
                if (L.live) ys[i + Q * p] = v;
                top = imax(top, fx_abs_hi(v));
            }
        }
        top >>= 20;
    } else {
        top = fx_slab_top<DIM, Q, SP>(ys, L.sub);
    }
    const FxBlock t{fx_cell_unit<DIM, Q, SP>(top, ys, L), 0};
    if (e0) fx_store_out<DIM, Q, SP>(u + cell0 * NL, reinterpret_cast<const double *>(Y), ncl * NL, L.lane);
    fx_to_block<DIM, Q, SP>(xs, ys, t.e, L);
    __syncwarp();
    fx_all_traces<DIM, Q, SP, USER>(tab, cst, xc, t, L, active, cell, tr,
                                    reinterpret_cast<const double *>(Y + L.c * G::C));
}

template <int DIM, int Q, int SP, bool USER>
__global__ void __launch_bounds__(FxGeo<DIM, Q, SP>::NW * 32)
    k_fx_project(const __grid_constant__ FxTab tab, const __grid_constant__ FxConst cst, double *u,
                 const double *__restrict__ e0, double *__restrict__ tr) {
    using G = FxGeo<DIM, Q, SP>;
    extern __shared__ __align__(16) long long smem_fx[];
    const int warp = threadIdx.x >> 5;
    const int64_t cell0 = (int64_t)blockIdx.x * G::CPB + warp * G::CW;
    if (cell0 >= cst.ncell) return;
    fx_project_body<DIM, Q, SP, USER>(tab, cst, smem_fx + warp * G::warp_words_project(), cell0, u, e0, tr);
}

template <int DIM, int Q, int SP>
__global__ void __launch_bounds__(FxGeo<DIM, Q, SP>::NW * 32)
    k_fx_project_batch(const __grid_constant__ FxTab tab, const BatchDG<double> *__restrict__ D,
                       const BlockMap *__restrict__ map, int nblocks, double *u, int with_e0) {
    using G = FxGeo<DIM, Q, SP>;
    extern __shared__ __align__(16) long long smem_fx[];
    __shared__ __align__(16) BatchDG<double> sd;
    const int warp = threadIdx.x >> 5;
    for (int k = blockIdx.x; k < nblocks; k += gridDim.x) {
        if (k != (int)blockIdx.x) __syncthreads();
        const BlockMap m = map[k];
        load_batch_desc(D + m.inst, &sd);
        const int64_t cell0 = (int64_t)m.cell0 + warp * G::CW;
        if (cell0 < sd.c.ncell)
            fx_project_body<DIM, Q, SP>(tab, sd.c, smem_fx + warp * G::warp_words_project(), cell0, u + sd.off * G::NL,
                                    with_e0 ? sd.e0 : nullptr, sd.tr[0]);
    }
}

template <typename K>
inline void fx_allow_smem(K *kernel, size_t bytes) {      // beside the static descriptor; no state kept
    if (bytes > 32 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Lanes per slab. On a small mesh a sub-core has at most one warp and that warp's own
// rate bounds the launch (q = 6: the same 49 us for 576 and 2744 cells), so the pencils
// of a slab go over SP lanes and a warp takes fewer cells (3D, q >= 5). Residual and four
// steps, one lane / split: q = 5, 576 cells 37 and 154 / 20 and 70 us, 2197 cells 37 and
// 154 / 35 and 109, 3375 cells 37 and 154 / 41 and 154; q = 6 576 cells 49 and 197 / 27 and
// 103, 2744 cells 50 and 204 / 70 and 239 (its second round of pencils is nearly empty);
// q = 7 512 cells 58 and 263 / 29 and 113, 2197 cells 62 and 271 / 58 and 251. In a batch the
// cells of all problems of a degree count (they share the launch).
template <int DIM, int Q>
constexpr int fx_split() {
    return DIM == 3 && Q >= 5 ? (Q == 5 ? 5 : 32 / Q) : 1;
}
template <int DIM, int Q>
inline bool fx_small(int64_t ncell) {
    return fx_split<DIM, Q>() > 1 && ncell <= (Q == 6 ? 1520 : 2432);
}

template <int DIM, int Q, int SP, int MODE>
cudaError_t fx_run_cells_of(const FxLevel &l, int flags, int mode, double *u, const double *b, const double *kappa,
                         const double *fd, const double *linv, const double *tri, double *tro, double *r,
                         double *corners, cudaStream_t s) {
    using G = FxGeo<DIM, Q, SP>;
    if (l.cst.ncell <= 0) return cudaSuccess;
    const size_t sm = G::bytes(MODE);
    fx_allow_smem(k_fx_cells<DIM, Q, SP, MODE>, sm);
    count_launches(1);
    k_fx_cells<DIM, Q, SP, MODE><<<(unsigned)((l.cst.ncell + G::CPB - 1) / G::CPB), G::NW * 32, sm, s>>>(
        l.tab, l.cst, flags, mode, u, b, kappa, fd, linv, tri, tro, r, corners);
    return cudaGetLastError();
}

template <int DIM, int Q, int MODE>
cudaError_t fx_run_cells(const FxLevel &l, int flags, int mode, double *u, const double *b, const double *kappa,
                         const double *fd, const double *linv, const double *tri, double *tro, double *r,
                         double *corners, cudaStream_t s) {
    if (fx_small<DIM, Q>(l.cst.ncell))
        return fx_run_cells_of<DIM, Q, fx_split<DIM, Q>(), MODE>(l, flags, mode, u, b, kappa, fd, linv, tri, tro, r,
                                                                 corners, s);
    return fx_run_cells_of<DIM, Q, 1, MODE>(l, flags, mode, u, b, kappa, fd, linv, tri, tro, r, corners, s);
}

// f(lanes per slab) of the work items of cpb cells (those of one lane where there is no split)
template <int DIM, int Q, typename F>
cudaError_t fx_batch_split(int cpb, F f) {
    constexpr int SP = fx_split<DIM, Q>();
    if (SP > 1 && cpb == FxGeo<DIM, Q, SP>::CPB) return f(std::integral_constant<int, SP>{});
    if (cpb == FxGeo<DIM, Q, 1>::CPB) return f(std::integral_constant<int, 1>{});
    return cudaErrorInvalidValue;
}

template <int DIM, int Q, int MODE>
cudaError_t fx_run_cells_batch(const FxTab &tab, int cpb, const BatchDG<double> *D, const BlockMap *map, int nblocks,
                               int flags, int mode, double *u, const double *b, double *r, int cur, cudaStream_t s) {
    if (nblocks <= 0) return cudaSuccess;
    return fx_batch_split<DIM, Q>(cpb, [&](auto split) -> cudaError_t {
        constexpr int SP = decltype(split)::value;
        using G = FxGeo<DIM, Q, SP>;
        const size_t sm = G::bytes(MODE);
        const auto fn = k_fx_cells_batch<DIM, Q, SP, MODE>;
        fx_allow_smem(fn, sm);
        count_launches(1);
        fn<<<persistent_grid((const void *)fn, G::NW * 32, sm, nblocks), G::NW * 32, sm, s>>>(tab, D, map, nblocks, flags,
                                                                                           mode, u, b, r, cur);
        return cudaGetLastError();
    });
}

template <int DIM, int Q>
cudaError_t FxRun<DIM, Q>::project(const FxLevel &l, bool user, double *u, const double *e0, double *tr, cudaStream_t s) {
    if (l.cst.ncell <= 0) return cudaSuccess;
    auto run = [&](auto split) -> cudaError_t {
        constexpr int SP = decltype(split)::value;
        using G = FxGeo<DIM, Q, SP>;
        const auto fn = user ? k_fx_project<DIM, Q, SP, true> : k_fx_project<DIM, Q, SP, false>;
        fx_allow_smem(fn, G::bytes_project());
        count_launches(1);
        fn<<<(unsigned)((l.cst.ncell + G::CPB - 1) / G::CPB), G::NW * 32, G::bytes_project(), s>>>(l.tab, l.cst, u, e0,
                                                                                                    tr);
        return cudaGetLastError();
    };
    if (fx_small<DIM, Q>(l.cst.ncell)) return run(std::integral_constant<int, fx_split<DIM, Q>()>{});
    return run(std::integral_constant<int, 1>{});
}
template <int DIM, int Q>
cudaError_t FxRun<DIM, Q>::smooth(const FxLevel &l, bool exact, int flags, double *u, const double *b,
                                  const double *kappa, const double *fd, const double *linv, const double *tri,
                                  double *tro, cudaStream_t s) {
    if (exact)
        return fx_run_cells<DIM, Q, FXM_SMOOTH>(l, flags, 0, u, b, kappa, fd, linv, tri, tro, nullptr, nullptr, s);
    return fx_run_cells<DIM, Q, FXM_SMOOTH_FULL>(l, flags, 0, u, b, kappa, fd, linv, tri, tro, nullptr, nullptr, s);
}
template <int DIM, int Q>
cudaError_t FxRun<DIM, Q>::residual(const FxLevel &l, bool user, int mode, const double *u, const double *b,
                                    const double *kappa, const double *tr, double *r, double *corners, cudaStream_t s) {
    if (user)
        return fx_run_cells<DIM, Q, FXM_RESIDUAL_USER>(l, 0, mode, const_cast<double *>(u), b, kappa, nullptr, nullptr,
                                                       tr, nullptr, r, corners, s);
    return fx_run_cells<DIM, Q, FXM_RESIDUAL>(l, 0, mode, const_cast<double *>(u), b, kappa, nullptr, nullptr, tr,
                                              nullptr, r, corners, s);
}
template <int DIM, int Q>
cudaError_t FxRun<DIM, Q>::project_batch(const FxTab &tab, int cpb, const BatchDG<double> *D, const BlockMap *map,
                                         int nblocks, double *u, int with_e0, cudaStream_t s) {
    if (nblocks <= 0) return cudaSuccess;
    return fx_batch_split<DIM, Q>(cpb, [&](auto split) -> cudaError_t {
        constexpr int SP = decltype(split)::value;
        using G = FxGeo<DIM, Q, SP>;
        const size_t sm = G::bytes_project();
        const auto fn = k_fx_project_batch<DIM, Q, SP>;
        fx_allow_smem(fn, sm);
        count_launches(1);
        fn<<<persistent_grid((const void *)fn, G::NW * 32, sm, nblocks), G::NW * 32, sm, s>>>(tab, D, map, nblocks, u,
                                                                                           with_e0);
        return cudaGetLastError();
    });
}
template <int DIM, int Q>
cudaError_t FxRun<DIM, Q>::smooth_batch(const FxTab &tab, int cpb, bool exact, const BatchDG<double> *D,
                                        const BlockMap *map, int nblocks, int flags, double *u, const double *b, int cur,
                                        cudaStream_t s) {
    if (exact)
        return fx_run_cells_batch<DIM, Q, FXM_SMOOTH>(tab, cpb, D, map, nblocks, flags, 0, u, b, nullptr, cur, s);
    return fx_run_cells_batch<DIM, Q, FXM_SMOOTH_FULL>(tab, cpb, D, map, nblocks, flags, 0, u, b, nullptr, cur, s);
}
template <int DIM, int Q>
cudaError_t FxRun<DIM, Q>::residual_batch(const FxTab &tab, int cpb, const BatchDG<double> *D, const BlockMap *map,
                                          int nblocks, int mode, const double *u, const double *b, double *r, int cur,
                                          cudaStream_t s) {
    return fx_run_cells_batch<DIM, Q, FXM_RESIDUAL>(tab, cpb, D, map, nblocks, 0, mode, const_cast<double *>(u), b, r,
                                                    cur, s);
}
template <int DIM, int Q>
int FxRun<DIM, Q>::cells_per_cta(int64_t ncell) {
    return fx_small<DIM, Q>(ncell) ? FxGeo<DIM, Q, fx_split<DIM, Q>()>::CPB : FxGeo<DIM, Q>::CPB;
}

}  // namespace dgmg
