// Prints results of the block fixed-point arithmetic (csrc/fx.cuh) on the host:
// reads "n, then n rows of k pairs a x" (hexadecimal floats), and prints per row the
// block's round trip of x and the sum of a x.
#include <cstdio>
#include <vector>

#include "fx.cuh"

using namespace dgmg;

int main() {
    int n = 0, k = 0;
    if (std::scanf("%d %d", &n, &k) != 2) return 1;
    for (int r = 0; r < n; ++r) {
        std::vector<double> a(k), x(k);
        int mx = 0;
        for (int i = 0; i < k; ++i) {
            if (std::scanf("%lf %lf", &a[i], &x[i]) != 2) return 1;
            mx = imax(mx, fx_abs_hi(x[i]));
        }
        const int ev = mx >> 20, e = fx_unit(ev);
        Acc s;
        acc_zero(s);
        for (int i = 0; i < k; ++i) {
            const long long t = fx_from(x[i], ev);
            std::printf("%a ", fx_to(t, e));
            mac(s, limb_of((long long)(a[i] * (double)(1ll << 59))), limb_of(t));   // |a| < 1: h below 2^27
        }
        std::printf("%a\n", fx_to(acc_value(s), e - 59 + 64));
    }
    return 0;
}
