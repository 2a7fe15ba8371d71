// The residual's weights on a grid of given spacings, as relative errors in units of 2^-53 of the products that the kernel
// forms: err[0..2] of 1/h_a^2 in Lap u, err[3..11] of (1 + delta/3) / h_a^2 in rows x, y, z, err[12..17] of
// 1 / (3 h_A h_B) in the mixed terms, err[18..20] of 1/h_a in At_ij.  Returns whether the spacings count as equal.
#include "mg_common.cuh"

extern "C" int outer_weight_errors(const double *h, int order, double *err)
{
    using namespace ctt;
    typedef long double L;
    Geo g{};
    for (int a = 0; a < 3; ++a) g.h[a] = h[a];
    const OuterInt o = make_outer_int(g, order);
    const int shu = order == 4 ? outer_shu<4>() : outer_shu<2>();
    const L c2 = order == 4 ? 1.5L : 1.0L, c1 = order == 4 ? 1.5L : 2.0L;
    auto rel = [](L v, L exact) { return (double)(fabsl(v / exact - 1) * 0x1p53L); };
    constexpr int pair[6][2] = {{0, 1}, {0, 2}, {1, 0}, {1, 2}, {2, 0}, {2, 1}};
    for (int a = 0; a < 3; ++a) {
        const L ih2 = 1 / ((L)h[a] * h[a]);
        err[a] = rel(c2 * ldexpl((L)o.w[0], -shu) * (o.iso ? 1 : ldexpl((L)o.wl[a], -62)), ih2);
        for (int A = 0; A < 3; ++A)
            err[3 + 3 * A + a] = rel(c2 * (L)o.w[10 + A] * (o.iso ? (A == a ? 4 : 3) : ldexpl((L)o.w3[A][a], -60)),
                                     ih2 * (A == a ? 4 : 3) / 3);
        err[18 + a] = rel(c1 * (L)o.ca * (o.iso ? 1 : ldexpl((L)o.ga[a], -63)), 1 / (L)h[a]);
    }
    for (int t = 0; t < 6; ++t)
        err[12 + t] = rel(c1 * c1 * (L)o.w[4 + t], 1 / (3 * (L)h[pair[t][0]] * (L)h[pair[t][1]]));
    return o.iso;
}
