// vkt_split_plan.h -- the weights and the error bound of the split evaluation of a separable
// filter (vkt_sep_split.cuh), prepared on the host in 64 bits.
#pragma once

#include <algorithm>
#include <cmath>

#include "vkt_internal.h"
#include "vkt_list_plan.h"

namespace vkt {

struct SplitPlan {
    float hi[3][VKT_MAX_FILTER_SIZE], lo[3][VKT_MAX_FILTER_SIZE];   // x, y, z: g = hi + lo
    float my, mz;                  // 1.5 * 2^23 * unit of h before the y and z passes
    float zg[VKT_MAX_FILTER_SIZE];  // the z weights times the mapping's scale (split in hi, lo)
    float whole, frac;             // code = whole + frac + H + L
    float tie;                     // 1/2 - the bound of the code's error
};

namespace split {

// g = hi + lo with hi a multiple of v, lo rounded to float32 (exact where g is a float32); false if sum|hi| * b (b in units of the input's grid)
// could exceed 24 bits of the product's grid
inline bool weights(const double* g, int k, double v, double b, float* hi, float* lo)
{
    double s = 0.0;
    for (int i = 0; i < k; ++i) {
        const double n = std::nearbyint(g[i] / v);
        s += std::fabs(n);
        hi[i] = static_cast<float>(n * v);
        lo[i] = static_cast<float>(g[i] - n * v);
    }
    return s * b <= 16777216.0;
}

}  // namespace split

// Fills `p` for the vectors g[0..2] of size k over a source of integer format sfmt (0: uint8,
// 1: uint16) and the uncentred code mapping a0 + a1 * sum (a0 = a0h + a0l, ...).  False if the
// evaluation does not suit the filter: weights that are not finite, results far outside the
// codes, flat regions on ties, or an error bound over 1/100 of a code (more than 1 in 50 voxels would be evaluated
// twice).
inline bool make_split_plan(SplitPlan& p, int k, const float* const g[3], int sfmt, float a0h,
                            float a0l, float a1h, float a1l)
{
    const double u = std::ldexp(1.0, -24);
    const double b0 = sfmt == vktDataFormatUint8 ? 128.0 : 32768.0;
    const double a1 = static_cast<double>(a1h) + a1l;
    if (!std::isfinite(a1)) return false;
    double w[3][VKT_MAX_FILTER_SIZE], sabs[3] = {0, 0, 0}, sum[3] = {0, 0, 0};
    for (int a = 0; a < 3; ++a)
        for (int i = 0; i < k; ++i) {
            w[a][i] = a == 2 ? a1 * g[a][i] : static_cast<double>(g[a][i]);
            if (!std::isfinite(w[a][i])) return false;
            // (tiny or huge weights: float32 products of the parts could leave the normal range)
            if (w[a][i] != 0.0 && (std::fabs(w[a][i]) < 1e-12 || std::fabs(w[a][i]) > 1e6)) return false;
            sabs[a] += std::fabs(w[a][i]);
            sum[a] += w[a][i];
        }
    const double a0 = static_cast<double>(a0h) + a0l + b0 * sum[0] * sum[1] * sum[2];
    if (!std::isfinite(a0)) return false;
    if (sabs[0] == 0.0 || sabs[1] == 0.0 || sabs[2] == 0.0) return false;
    // reach: the largest code any pass could give
    const double reach = std::fabs(a0) + sabs[0] * sabs[1] * sabs[2] * b0;
    if (!(reach < 2097152.0)) return false;

    double bound = b0, err = 0.0, bl = 0.0;   // of a pass's input: |value|, error; |L| of its output
    for (int a = 0; a < 3; ++a) {
        double best = -1.0, best_u = 1.0, best_v = 1.0, best_bl = 0.0;
        // the unit of h: 1 (the codes themselves) for the x pass, a power of two for the others
        const int top = static_cast<int>(std::ceil(std::log2(bound))) + 1;
        for (int eu = a == 0 ? 0 : top - 21; eu <= (a == 0 ? 0 : top - 5); ++eu) {
            const double unit = std::ldexp(1.0, eu);
            const double bh = a == 0 ? bound : bound + unit;            // |h|
            const double rest = a == 0 ? 0.0 : 0.5 * unit + 2.0 * u * bound;   // |l|
            double v = std::ldexp(1.0, static_cast<int>(std::floor(std::log2(sabs[a] * bh / unit))) - 24);
            float hi[VKT_MAX_FILTER_SIZE], lo[VKT_MAX_FILTER_SIZE];
            while (!split::weights(w[a], k, v, bh / unit, hi, lo)) v *= 2.0;
            // the roundings of L: a running sum of wl h (and g l) terms
            double part = 0.0, roundings = 0.0;
            for (int i = 0; i < k; ++i) {
                part += std::fabs(static_cast<double>(lo[i])) * bh;
                roundings += part;
                if (a > 0) {
                    part += std::fabs(w[a][i]) * rest;
                    roundings += part;
                }
            }
            // (u * part: lo and the scaled z weights are rounded to float32)
            const double e = sabs[a] * (err + u * rest) + u * roundings + u * part;
            if (best < 0.0 || e < best) {
                best = e;
                best_u = unit;
                best_v = v;
                best_bl = part;
            }
        }
        split::weights(w[a], k, best_v, 1.0, p.hi[a], p.lo[a]);
        if (a == 1) p.my = static_cast<float>(1.5 * 8388608.0 * best_u);
        if (a == 2) p.mz = static_cast<float>(1.5 * 8388608.0 * best_u);
        err = best;
        bl = best_bl;
        bound = bound * sabs[a] + err;
    }
    for (int i = 0; i < k; ++i) p.zg[i] = static_cast<float>(w[2][i]);
    p.whole = static_cast<float>(std::nearbyint(a0));
    p.frac = static_cast<float>(a0 - static_cast<double>(p.whole));
    // the roundings of frac, L + frac and the sum with H's remainder, and what the Dot2 evaluation
    // itself may be off (errors of second order, below 1e-7 of a 16-bit code)
    const double e = err + 3.0 * u * (bl + 2.0) + 1e-6 * std::max(1.0, reach / 65536.0);
    p.tie = static_cast<float>(0.5 - e * 1.0001) * (1.f - 1.2e-7f);
    const double slope = sum[0] * sum[1] * sum[2];
    return e < 0.01 && !flat_field_ties(a0 - b0 * slope, slope, sfmt, e);
}

}  // namespace vkt
