// vkt_list_plan.h -- the weights and the error bound of the listed modes of the direct kernel
// (vkt_direct.cuh), prepared on the host in 64 bits.
#pragma once

#include <algorithm>
#include <cmath>

#include "vkt_internal.h"

namespace vkt {

struct ListPlan {
    bool pair;                     // high and low weights, else one float32 weight
    bool exact;                    // every sum is exact: ties are told apart, none is listed
    float w[VKT_MAX_FILTER_SIZE * VKT_MAX_FILTER_SIZE * VKT_MAX_FILTER_SIZE];
    float l[VKT_MAX_FILTER_SIZE * VKT_MAX_FILTER_SIZE * VKT_MAX_FILTER_SIZE];
    float whole, frac;             // code = whole + frac + H (+ L)
    float tie;                     // 1/2 less the bound of the code's error
};

// Whether a field of one code everywhere (a scan's background, a saturated region) maps onto a
// rounding tie, within `e`, for any of a few codes at the ends of the range: whole regions would
// then be listed, which costs more than Dot2 does.
inline bool flat_field_ties(double a0, double slope, int sfmt, double e)
{
    const double top = sfmt == vktDataFormatUint8 ? 255.0 : 65535.0;
    for (double q : {0.0, 1.0, 2.0, 3.0, top - 1.0, top}) {
        const double v = a0 + slope * q;
        if (std::fabs(std::fabs(v - std::nearbyint(v)) - 0.5) <= e) return true;
    }
    return false;
}

// The plan of the k^3 weights g over a source of integer format sfmt into the codes
// a0 + a1 * sum (a0 = a0h + a0l, ...).  One float32 weight per tap where at most about 1 voxel
// in 100 lies within its error bound of a tie (a uint8 destination up to k = 7 or so), else the
// pair where at most 1 in 16 does; 256 x 256 x 200, Dot2 / listed: uint8 k = 5 642 / 100 us,
// k = 7 1903 / 310; uint16 k = 3 185 / 57, k = 5 642 / 231 (the pair, 1 voxel in 33 listed), k = 7
// 2017 / 1769 with 1 in 4 listed and 94 / 141 on 64^3, so that stays with Dot2.  False
// if neither, if flat regions lie on ties, or if the weights are not finite or reach far outside
// the codes.  Weights and offset that are multiples of a power of two (a Laplacian into a
// symmetric range puts half of all voxels on ties) need no bound: their sums are exact.
// The bound of a chain of FMAs in tap order: every rounding is at most 2^-24 of the partial sum
// it rounds, and that is at most the sum of the |terms| so far.
inline bool make_list_plan(ListPlan& p, int k, const float* g, int sfmt, float a0h, float a0l,
                           float a1h, float a1l)
{
    const double u = std::ldexp(1.0, -24);
    const double b = sfmt == vktDataFormatUint8 ? 128.0 : 32768.0;
    const int n = k * k * k;
    const double a1 = static_cast<double>(a1h) + a1l;
    double sabs = 0.0, sum = 0.0, prefix = 0.0;
    for (int i = 0; i < n; ++i) {
        const double w = a1 * g[i];
        // (tiny or huge weights: products of the parts could leave float32's normal range)
        if (!std::isfinite(w) || (w != 0.0 && (std::fabs(w) < 1e-12 || std::fabs(w) > 1e6))) return false;
        sabs += std::fabs(w);
        sum += w;
        prefix += sabs;
    }
    const double a0 = static_cast<double>(a0h) + a0l + b * sum;
    const double reach = std::fabs(a0) + sabs * b;
    if (!(reach < 2097152.0) || sabs == 0.0) return false;
    // the epilogue's roundings, and what Dot2 itself may be off: (n u)^2 of the absolute sum, and
    // its mapping's rounding
    const double nu = n * u;
    const double own = 3.0 * u * 2.0 + 1.1 * nu * nu * 2.0 * sabs * b + 1e-6 * std::max(1.0, reach / 65536.0);
    p.whole = static_cast<float>(std::nearbyint(a0));
    p.frac = static_cast<float>(a0 - static_cast<double>(p.whole));
    // the finest unit v that sums of 24 bits leave room for
    double v = std::ldexp(1.0, static_cast<int>(std::floor(std::log2(sabs * b))) - 24), off = 0.0;
    for (;; v *= 2.0) {
        double s = 0.0;
        off = 0.0;
        for (int i = 0; i < n; ++i) {
            const double m = std::nearbyint(a1 * g[i] / v);
            s += std::fabs(m);
            off += std::fabs(a1 * g[i] - m * v);
        }
        if (s * b <= 16777216.0) break;
    }
    const double dyadic = std::nearbyint((a0 - p.whole) * 4096.0) / 4096.0;
    p.exact = off * b < 2e-9 && std::fabs(a0 - p.whole - dyadic) < 1e-9;
    if (p.exact) {
        // (Dot2 sees what is off as far less than the last bit at a tie)
        for (int i = 0; i < n; ++i) p.w[i] = static_cast<float>(std::nearbyint(a1 * g[i] / v) * v);
        p.pair = false;
        p.frac = static_cast<float>(dyadic);
        p.tie = 1.f;   // never reached
        return true;
    }
    double e = u * b * (prefix + sabs) + own;
    p.pair = e >= 0.005;
    if (!p.pair) {
        for (int i = 0; i < n; ++i) p.w[i] = static_cast<float>(a1 * g[i]);
    } else {
        // H exact: sum |w| b is at most 2^24 units v
        double low = 0.0, roundings = 0.0;
        for (int i = 0; i < n; ++i) {
            const double h = std::nearbyint(a1 * g[i] / v) * v;
            p.w[i] = static_cast<float>(h);
            p.l[i] = static_cast<float>(a1 * g[i] - h);
            low += std::fabs(a1 * g[i] - h);
            roundings += low;
        }
        e = u * b * (roundings + low) + 2.0 * u * b * low + own;
    }
    p.tie = static_cast<float>(0.5 - e * 1.0001) * (1.f - 1.2e-7f);
    return e < 0.03 && !flat_field_ties(a0 - b * sum, sum, sfmt, e);
}

}  // namespace vkt
