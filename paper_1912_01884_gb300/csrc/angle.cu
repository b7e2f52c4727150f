// The bend-angle windows of Sec. 2.3 (host side).
#include <cmath>

#include "chain.cuh"

namespace fhtdp {

// Fig. 5: a link of displacement d over n rows has inclination atan(d / n);
// the bend angle between links d and e is |atan(e / n) - atan(d / n)|.  As
// atan is increasing, the admissible e for one d form an interval (the
// union of the ranges of Eqs. 6 and 7), and both of its ends are
// non-decreasing in d, so one sweep with two pointers finds every interval.
// The comparison is the definition itself, evaluated in double.
bool make_angle_table(int n, double gamma, WindowTable *t) {
    if (!(gamma >= 0.0) || !std::isfinite(gamma) || n < 1 || 2 * n - 1 > kMaxD) return false;
    const int D = 2 * n - 1;
    double a[kMaxD];
    for (int i = 0; i < D; ++i) a[i] = std::atan((double)(i - (n - 1)) / n);
    int lo = 0, hi = 0;
    for (int i = 0; i < D; ++i) {
        while (a[i] - a[lo] > gamma) ++lo;
        if (hi < i) hi = i;
        while (hi + 1 < D && a[hi + 1] - a[i] <= gamma) ++hi;
        t->lo[i] = (int16_t)(lo - (n - 1));
        t->hi[i] = (int16_t)(hi - (n - 1));
    }
    for (int i = D; i < kMaxD; ++i) t->lo[i] = t->hi[i] = 0;
    t->n = n;
    return true;
}

// Subproblem 3 and the main problem run on the chain (chain.cu): the smoothed
// rows, the band FHTs and the DP with the window table.
size_t angle_workspace_bytes(const Shape &s) { return chain_layout(s, true).total; }

}  // namespace fhtdp
