// Host side of the block fixed-point FP64 kernels (fx.cuh): the limbs of the
// reference element's tables and of a level's mesh-dependent vectors, formed in
// extended precision from the FP64 reference element.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "internal.h"

namespace dgmg {

namespace {

using R = long double;

// exponent e with bound / 2^e < 2^bits
int unit_for(R bound, int bits) {
    int e = 0;
    std::frexp(bound, &e);                        // bound < 2^e
    return bound > 0 ? e - bits : 0;
}
Limb limb(R v, int e) { return limb_of((long long)std::llrint(std::ldexp(v, -e))); }

// largest row sum of magnitudes of q x q matrices added up
R row_sum(int q, const std::vector<const std::vector<R> *> &ms) {
    R top = 0;
    for (int i = 0; i < q; ++i) {
        R s = 0;
        for (const auto *m : ms)
            for (int j = 0; j < q; ++j) s += std::fabs((*m)[i * q + j]);
        top = std::max(top, s);
    }
    return top;
}
R largest(const std::vector<R> &v) {
    R t = 0;
    for (R x : v) t = std::max(t, std::fabs(x));
    return t;
}
R total(const std::vector<R> &v) {
    R t = 0;
    for (R x : v) t += std::fabs(x);
    return t;
}

// inverse of a small matrix by Gauss-Jordan elimination with column pivoting
std::vector<R> inverse(int q, std::vector<R> A) {
    std::vector<R> B(q * q, 0);
    for (int i = 0; i < q; ++i) B[i * q + i] = 1;
    for (int c = 0; c < q; ++c) {
        int p = c;
        for (int i = c + 1; i < q; ++i)
            if (std::fabs(A[i * q + c]) > std::fabs(A[p * q + c])) p = i;
        for (int j = 0; j < q; ++j) {
            std::swap(A[c * q + j], A[p * q + j]);
            std::swap(B[c * q + j], B[p * q + j]);
        }
        const R d = A[c * q + c];
        for (int j = 0; j < q; ++j) {
            A[c * q + j] /= d;
            B[c * q + j] /= d;
        }
        for (int i = 0; i < q; ++i) {
            if (i == c) continue;
            const R f = A[i * q + c];
            for (int j = 0; j < q; ++j) {
                A[i * q + j] -= f * A[c * q + j];
                B[i * q + j] -= f * B[c * q + j];
            }
        }
    }
    return B;
}

std::vector<R> times(int q, const std::vector<R> &A, const std::vector<double> &v) {
    const int cols = (int)v.size() / q;
    std::vector<R> out((size_t)q * cols, 0);
    for (int i = 0; i < q; ++i)
        for (int j = 0; j < cols; ++j)
            for (int k = 0; k < q; ++k) out[i * cols + j] += A[i * q + k] * (R)v[k * cols + j];
    return out;
}

// The magnitudes the kernels count on (fx.cuh, mac): the h of a row of a matrix
// sum to at most 2^31, those of a single factor are at most 2^30. The mass, and the
// eigenvectors (k_fx_factors), whose passes follow one another in the smoothing step, use
// all of it (pass_unit): with a bit less a step on 40 x 2 x 2 cells, p = 3, was off by up to
// 1.2e-14 of a cell's largest value (FP64 pipe 4.6e-15, now 5.6e-15), and by up to 1.7e-14
// from b = A u (7.4e-15, 1.0e-14).
constexpr int ROW_BITS = 62, ONE_BITS = 61, PASS_BITS = 63;
int pass_unit(R bound) { return unit_for(bound * (1 + 0x1p-30L), PASS_BITS); }   // (an h stays below 2^31)

// What a level takes from its element: the tables, and M^-1 of the end values.
struct Element {
    FxTab tab;
    std::vector<R> m0, mp;
};

Element make_element(const RefElem1D &re, int penalty_p) {
    Element el;
    FxTab &tab = el.tab;
    std::memset(&tab, 0, sizeof(tab));
    const int q = re.q;
    tab.gl = re.basis == DGMG_BASIS_GL ? 1 : 0;
    const std::vector<R> M(re.M.begin(), re.M.end()), Mi = inverse(q, M);
    const std::vector<R> K = times(q, Mi, re.K);
    const std::vector<R> m0 = times(q, Mi, re.e0), mp = times(q, Mi, re.ep), d0 = times(q, Mi, re.d0),
                         dp = times(q, Mi, re.dp);
    const R pen = (R)penalty_p * (penalty_p + 1);
    std::vector<R> L[2], Rt[2];
    for (int w = 0; w < 2; ++w) {
        const R wt = w ? 1.0L : 0.5L;
        L[w].resize(q * q);
        Rt[w].resize(q * q);
        for (int i = 0; i < q; ++i)
            for (int j = 0; j < q; ++j) {
                L[w][i * q + j] = wt * (m0[i] * re.d0[j] + d0[i] * re.e0[j]) + pen * m0[i] * re.e0[j];
                Rt[w][i * q + j] = -wt * (mp[i] * re.dp[j] + dp[i] * re.ep[j]) + pen * mp[i] * re.ep[j];
            }
    }
    tab.eM = pass_unit(row_sum(q, {&M}));
    R rows = 0;
    for (int w = 0; w < 4; ++w) rows = std::max(rows, row_sum(q, {&K, &L[w & 1], &Rt[w >> 1]}));
    tab.eD = unit_for(rows, ROW_BITS);
    for (int i = 0; i < q * q; ++i) {
        tab.M[i] = limb(M[i], tab.eM);
        tab.K[i] = limb(K[i], tab.eD);
        for (int w = 0; w < 2; ++w) {
            tab.L[w][i] = limb(L[w][i], tab.eD);
            tab.R[w][i] = limb(Rt[w][i], tab.eD);
        }
    }
    std::vector<R> g(2 * q), hat(2 * q), v(2 * q);
    for (int i = 0; i < q; ++i) {
        g[i] = -d0[i] / 2 - pen * m0[i];
        g[q + i] = dp[i] / 2 - pen * mp[i];
        hat[i] = (1.0L - (R)re.nodes[i]) / 2;
        hat[q + i] = (1.0L + (R)re.nodes[i]) / 2;
        v[i] = re.e0[i];
        v[q + i] = re.ep[i];
    }
    tab.eG = unit_for(largest(g), ONE_BITS);
    tab.eHat = unit_for(total(hat), ROW_BITS);
    tab.eV = unit_for(total(v), ROW_BITS);
    for (int s = 0; s < 2; ++s)
        for (int i = 0; i < q; ++i) {
            tab.cG[s][i] = limb(g[s * q + i], tab.eG);
            tab.hat[s][i] = limb(hat[s * q + i], tab.eHat);
            tab.v[s][i] = limb(v[s * q + i], tab.eV);
        }
    el.m0 = m0;
    el.mp = mp;
    return el;
}

// One per (nodes, basis, penalty degree), at most 7 x 2 x 6: formed once in the
// process (extended precision is software on the host of a GB300: 0.4 ms each).
const Element &element(const RefElem1D &re, int penalty_p) {
    static std::mutex mu;
    static std::map<std::tuple<int, int, int>, Element> all;   // nodes of a map stay where they are
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_tuple(re.q, re.basis, penalty_p);
    auto it = all.find(key);
    if (it == all.end()) it = all.emplace(key, make_element(re, penalty_p)).first;
    return it->second;
}

}  // namespace

void fx_tables(const RefElem1D &re, int penalty_p, FxTab &tab) { tab = element(re, penalty_p).tab; }

void fx_level(const RefElem1D &re, int penalty_p, int dim, const int *n, int64_t ncell, double keep, FxConst &cst) {
    std::memset(&cst, 0, sizeof(cst));
    const int q = re.q;
    const Element &el = element(re, penalty_p);
    for (int a = 0; a < 3; ++a) cst.n[a] = n[a];
    cst.ncell = ncell;
    R vol = 1;
    for (int a = 0; a < dim; ++a) vol *= 0.5L / n[a];
    for (int a = 0; a < dim; ++a) {
        const R h = 1.0L / n[a];
        cst.sa[a] = (double)(vol * 4 / (h * h));
        std::vector<R> c(2 * q), d(2 * q);
        for (int i = 0; i < q; ++i) {
            c[i] = h / 4 * el.m0[i];
            c[q + i] = -h / 4 * el.mp[i];
            d[i] = 2 / h * (R)re.d0[i];
            d[q + i] = 2 / h * (R)re.dp[i];
        }
        cst.eH[a] = unit_for(largest(c), ONE_BITS);
        cst.eT[a] = unit_for(total(d), ROW_BITS);
        for (int s = 0; s < 2; ++s)
            for (int i = 0; i < q; ++i) {
                cst.cH[a][s][i] = limb(c[s * q + i], cst.eH[a]);
                cst.dt[a][s][i] = limb(d[s * q + i], cst.eT[a]);
            }
    }
    cst.keep = keep;
}

}  // namespace dgmg
