// Block fixed-point arithmetic for the FP64 kernels of the DG levels.
//
// GB300 issues 1.6 FP64 multiply-adds per SM and clock (dgmg_fma_peak), but 30 of
// the integer 32 x 32 + 64 bit multiply-add (a loop of independent products). A
// product of two 60-bit numbers kept as two 32-bit limbs takes three of them (the
// product of the low limbs is below the result's last place): 10 multiply-adds per
// SM and clock, six times the FP64 pipe, with a longer significand.
//
// A block of numbers (the tensor of a cell) shares one exponent: value = t 2^e with a
// 64-bit integer t, |t| < 2^60. After every matrix the block is shifted left to use
// all 60 bits, so a stage loses about 2^-58 of the block's largest value, where FP64
// loses 2^-53 of every product: norm by norm, cell by cell, the sums are at least as
// exact, but a value far below its block's largest holds fewer bits than FP64 would keep.
// So the vectors stay FP64 and are added to and subtracted from node by node (dg_fx.cuh),
// and the table of the block inverses, whose entries span the cell's eigenvalues, keeps an
// exponent per entry (fx_scaled). Largest errors against a 64-bit reference, FP64 pipe
// kernels before / these: operator p = 4, 64 x 60 x 57 cells 2.4e-15 / 2.4e-15; residual p = 6
// GL, 243 x 241 cells 4.3e-15 / 4.1e-15; four smoothing steps p = 3, 33 x 31 x 32 cells 2.5e-15
// / 2.5e-15, p = 4, 729^2 cells 8.6e-16 / 8.3e-16 (near the reference's own rounding); V-cycles
// 16^2 p = 2 7.1e-16 / 7.9e-16, 23 x 17 x 20 p = 2 9.9e-16 / 1.2e-15.
//
// An input that is not finite marks its block (e >= FX_BAD), and every value
// computed from a marked block is output as NaN. Results above the normal range are
// output as infinity, below it as subnormal numbers, and subnormal inputs count as what
// they are.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace dgmg {

constexpr int FX_BAD = 1 << 19;         // exponents from here on: not finite
constexpr int FX_NONE = -(1 << 19);     // exponent of a block without values

// h 2^32 + l with a signed low limb
struct Limb {
    int h, l;
};

#define FX_HD __host__ __device__ __forceinline__

FX_HD Limb limb_of(long long t) {
    Limb x;
    x.l = (int)(unsigned)t;
    x.h = (int)(t >> 32) + (int)((unsigned)x.l >> 31);
    return x;
}

// Sum of products of limbs: hh counts 2^64, m counts 2^32 (half a unit of hh to
// start with, so that the value is rounded, not cut). With |x| < 2^60 and the h of
// the n <= 7 factors summing to at most 2^31 in magnitude both stay below 2^63
// (|hh| <= 2^59, |m| <= 2^62 + 7 2^59 + 2^31).
struct Acc {
    long long hh, m;
};
FX_HD void acc_zero(Acc &s) {
    s.hh = 0;
    s.m = 1ll << 31;
}
// c + a b. On the device as a carry pair, which becomes the one wide multiply-add it
// is; mad.wide lets the assembler rebalance a sum of products into separate 64-bit
// adds (12 more instructions per four products, by the opcode counters). The low word
// is written before the factors are read again: it shares no register with them.
FX_HD long long mad_wide(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
    unsigned lo = (unsigned)c, hi = (unsigned)((unsigned long long)c >> 32);
    asm("mad.lo.cc.s32 %0, %2, %3, %0;\n\tmadc.hi.s32 %1, %2, %3, %1;" : "+&r"(lo), "+r"(hi) : "r"(a), "r"(b));
    return (long long)((unsigned long long)hi << 32 | lo);
#else
    return c + (long long)a * b;
#endif
}
FX_HD void mac(Acc &s, Limb a, Limb x) {
    s.hh = mad_wide(a.h, x.h, s.hh);
    s.m = mad_wide(a.h, x.l, s.m);
    s.m = mad_wide(a.l, x.h, s.m);
}
// the sum as a block value, its unit 2^64 times the product of the units
FX_HD long long acc_value(const Acc &s) { return mad_wide((int)(s.m >> 32), 1, s.hh); }

FX_HD int hi_word(double v) {
#ifdef __CUDA_ARCH__
    return __double2hiint(v);
#else
    union { double d; int64_t i; } x = {v};
    return (int)(x.i >> 32);
#endif
}
FX_HD int lo_word(double v) {
#ifdef __CUDA_ARCH__
    return __double2loint(v);
#else
    union { double d; int64_t i; } x = {v};
    return (int)x.i;
#endif
}
FX_HD double from_words(int hi, int lo) {
#ifdef __CUDA_ARCH__
    return __hiloint2double(hi, lo);
#else
    union { int64_t i; double d; } x = {(int64_t)(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo)};
    return x.d;
#endif
}
FX_HD int clz32(int v) {
#ifdef __CUDA_ARCH__
    return __clz(v);
#else
    return v == 0 ? 32 : __builtin_clz((unsigned)v);
#endif
}
FX_HD int imax(int a, int b) { return a > b ? a : b; }
FX_HD int imin(int a, int b) { return a < b ? a : b; }

// Largest biased exponent of a block of FP64 values: mx over fx_abs_hi, >> 20.
FX_HD int fx_abs_hi(double v) { return hi_word(v) & 0x7fffffff; }
FX_HD bool fx_some(double v) { return (fx_abs_hi(v) | lo_word(v)) != 0; }   // not 0

// FP64 value as a block value of unit 2^(ev - FX_UNIT); ev >= its biased exponent, and at
// least FX_LOW (subnormal values are below the unit then).
constexpr int FX_UNIT = 1023 + 59, FX_LOW = 61;
FX_HD long long fx_from(double v, int ev) {
    const int hi = hi_word(v), lo = lo_word(v);
    const int e = (hi >> 20) & 0x7ff, d = imin(ev - e, 63);      // the significand ends at bit 59: d >= 60 gives 0
    const unsigned top = (unsigned)(hi & 0xfffff) | (e ? 0x100000u : 0u);
    const long long m = (long long)((((unsigned long long)top << 32 | (unsigned)lo) << 7) >> (d & 63));
    const long long s = hi >> 31;
    return (m ^ s) - s;
}
// The same for every ev, below 1 (a block of subnormal values) too.
FX_HD long long fx_from_any(double v, int ev) {
    const int hi = hi_word(v), lo = lo_word(v), e = (hi >> 20) & 0x7ff, d = ev - imax(e, 1);
    const unsigned top = (unsigned)(hi & 0xfffff) | (e ? 0x100000u : 0u);
    const unsigned long long x = ((unsigned long long)top << 32 | (unsigned)lo) << 7;
    const long long m = (long long)(d >= 0 ? x >> imin(d, 63) : x << imin(-d, 63)), s = hi >> 31;
    return (m ^ s) - s;
}
// exponent (unit) of a block whose largest biased exponent is ev
FX_HD int fx_unit(int ev) { return ev >= 2047 ? 2 * FX_BAD : (ev <= 0 ? FX_NONE : ev - FX_UNIT); }

// Block value t 2^e as FP64, rounded to nearest (ties away from zero). SAFE: every value of
// the block is 0 or in the normal range (fx_safe), as nearly always: without the look at the
// range, which costs more than its instructions (operator 64 x 60 x 57 p = 4 1142 us without
// subnormal results, 1169 with their code behind every value, 1131 with the look by blocks).
FX_HD bool fx_safe(int e) { return (unsigned)(e + 1022) <= 1900u; }
template <bool SAFE = false>
FX_HD double fx_to(long long t, int e) {
    const int s = (int)(t >> 63);
    unsigned long long a = (unsigned long long)((t ^ (long long)s) - (long long)s);
    if ((a >> 32) == 0) {                        // rare: far below the block's largest value
        a <<= 31;
        e -= 31;
    }
    const int n = clz32((int)(a >> 32)) - 1;     // top bit to bit 62
    a = (a << (n & 63)) + 512;
    const int be = e - n + 62 + 1023;            // biased exponent of bit 62
    int hi = ((int)(a >> 42) + ((be - 1) << 20)) | (s & (int)0x80000000), lo = (int)(unsigned)(a >> 10);
    if (t == 0) hi = lo = 0;
    if (!SAFE && ((unsigned)(be - 1) >= 2046u || (t == 0 && e >= FX_BAD - 64))) {
        hi = 0x7ff00000 | (s & (int)0x80000000);
        lo = 0;
        if (t == 0 || be < 1) {                  // subnormal: fewer bits of the significand
            const int d = imin(11 - be, 63);     // (63: half the least number)
            a = t == 0 || be < -52 ? 0 : (a - 512 + (1ull << (d - 1))) >> d;
            hi = (int)(a >> 32) | (s & (int)0x80000000);
            lo = (int)(unsigned)a;
        }
        if (e >= FX_BAD - 64) hi = 0x7ff80000, lo = 0;
    }
    return from_words(hi, lo);
}

// Arithmetic right shift by d >= 0 of any size.
FX_HD long long fx_shr(long long t, int d) { return t >> imin(d, 63); }

// Block values times numbers of any spread, as a block again. Where the largest value
// meets the smallest number (the modes of a cell and the inverses of their eigenvalues)
// the products are far below the product of the two largest, and one unit for the numbers
// and one for the bound on the products would cost the ratio's bits: a smoothing step from
// b = A u had two to six times the FP64 pipe's error. So every number has its exponent and
// all of its 53 bits, a product is formed from both factors at full length, and the
// block's unit follows the largest product: fx_scaled_below per value, the least of them
// to fx_scaled. (A running maximum of the negated sums came out wrong from CUDA 13.0's
// assembler wherever it was not unrolled in full: the sums are kept positive.)
//
// A number of the table as a word: the limbs of its significand (top bit 61, the low 9
// zero), in those 9 bits of the low limb the exponent below the table's.
constexpr int FX_BELOW = 511;
FX_HD long long fx_table_word(double w, int base) {          // |w| < 2^(base + 1)
    int e = 0;
    const double f = frexp(w, &e);
    const int below = base - (e - 1);
    if (!(f != 0.0) || below > FX_BELOW) return FX_BELOW;    // (and what is not finite: the table is marked)
    const Limb x = limb_of((long long)ldexp(f, 62));
    return (long long)((unsigned long long)(unsigned)x.h << 32 | ((unsigned)x.l | (unsigned)below));
}
FX_HD int fx_lead(long long t) {                             // the sign's leading copies (at most 32)
    const int h = (int)(t >> 32);
    return clz32(h ^ (h >> 31));
}
FX_HD int fx_scaled_below(long long t, long long w) { return ((int)w & FX_BELOW) + fx_lead(t); }
constexpr int FX_SCALED_MOST = FX_BELOW + 32;
// |t| < 2^60; the result below 2^58, in units of 2^(e + base + FX_SCALED - least) for a t of unit 2^e
constexpr int FX_SCALED = 64 - 61 + 4;
FX_HD long long fx_scaled(long long t, long long w, int least) {
    const int lead = fx_lead(t), below = (int)w & FX_BELOW;
    Acc s;
    acc_zero(s);
    mac(s, Limb{(int)(w >> 32), (int)w & ~FX_BELOW}, limb_of(t << ((lead - 4) & 63)));
    return acc_value(s) >> imin(below + lead - least, 63);
}

constexpr int FXQ = 7;                  // most nodes per axis

// Matrices and vectors of the reference element, packed row-major with the q
// nodes of the level (entries of one group share an exponent). With M^ the mass
// on [-1,1] and m0 = M^^-1 e0, md0 = M^^-1 d0 (end values and derivatives at the
// low end; mp, mdp at the high end):
//   M   mass;   K  M^^-1 K^;
//   L[w], R[w]  the cell's own face terms in M^^-1, low and high face, interior
//               (w = 0: weight 1/2) and boundary (w = 1: weight 1):
//               w (m0 d0^T + md0 e0^T) + p(p+1) m0 e0^T,
//               -w (mp dp^T + mdp ep^T) + p(p+1) mp ep^T;
//   cG[side]    coefficients of the neighbour's value trace:
//               -md0/2 - p(p+1) m0, mdp/2 - p(p+1) mp;
//   hat, v      hat values at the nodes; end values of the basis (GL).
struct FxTab {
    Limb M[FXQ * FXQ], K[FXQ * FXQ], L[2][FXQ * FXQ], R[2][FXQ * FXQ];
    Limb cG[2][FXQ], hat[2][FXQ], v[2][FXQ];
    int eM, eD, eG, eHat, eV;
    int gl;
};

// Data of one DG level: mesh, scales, and the vectors that depend on the cell
// width. sa[a] = (product of h/2 over the axes) 4 / h_a^2 scales kappa to the
// coefficient of axis a's terms between the mass inverse and the masses; kfac
// holds the facet coefficients times sa of their axis.
struct FxConst {
    int n[3];
    int64_t ncell;
    double sa[3];
    Limb cH[3][2][FXQ], dt[3][2][FXQ];  // neighbour's derivative trace; derivatives at the cell's ends
    int eH[3], eT[3];
    double keep;                        // 1 - omega (exact blocks) or 1
    const double *kfac;                 // [cell][2 axis + side], 0 on the boundary
};

}  // namespace dgmg
