// vkt_sep_split.cuh -- one brick of the fused separable filter from an integer source into
// an integer destination whose codes an FP32 evaluation could flip (separable_needs_comp).
//
// The codes must be those of the compensated (Dot2) evaluation, whose three passes cost about
// 160 flops per voxel at k = 5.  Here a voxel is first evaluated as a pair H + L:
//   - the source codes are centred (v = q - 2^(bits-1), exact), and every weight is split
//     g = wh + wl, wh a multiple of a power of two chosen so that sum(wh * v) is exact in
//     float32 (at most 24 bits: all partial sums are multiples of one unit and below 2^24
//     of it);
//   - x pass: H = sum(wh v) exact, L = sum(wl v), small, so its rounding is small;
//   - between the passes the pair is rounded to h (a multiple of a unit U, by adding and
//     subtracting 1.5 * 2^23 U) and the rest l = (H - h) + L, and the next pass takes
//     H = sum(wh h) exact, L = sum(wl h + g l);
//   - the scale of the value mapping is folded into the z weights and the centring into its
//     offset, so the code is the nearest integer of A + f + H + L, A an integer: H is rounded
//     to an integer (by adding and subtracting 1.5 * 2^23), then what that leaves plus L + f,
//     and the last remainder says how far the nearest tie is.
// The host bounds the error of that value (split_plan): about 1e-5 of a 16-bit code for a
// normalised Gaussian.  A voxel whose value lies nearer than that bound to a rounding tie is
// put on a list in shared memory and evaluated again with the Dot2 sequence of brick_comp, a
// thread per voxel, so the codes are the Dot2 codes bit for bit; about 1 in 10^4 voxels is.
// (Evaluating the listed voxels where they occur would leave 31 lanes waiting each time.)
// 8 FMAs per tap of the three passes instead of 32 flops: 94 instructions per voxel at k = 5
// where Dot2 has 200.  512 x 512 x 256 uint16 -> uint16, k = 5: 635 -> 304 us (0.88 TB/s); bound
// by latency at 16 warps per SM (issue 47 %, barrier and fixed-latency stalls), of which the
// listed voxels take 17 us (45 us with a thread per voxel also for short lists).
#pragma once

#include "vkt_sep_brick.cuh"
#include "vkt_split_plan.h"
#include "vkt_window.cuh"

namespace vkt {
namespace sep {

// The split weights of one filter for one (source, destination) pair; see split_plan.
template <int K>
struct SplitW {
    float2 xh[K], xl[K];           // x pass: source codes are exact (each weight twice: the
    float2 yh[K], yl[K], yw[K];    // operands of the packed FMAs)
    float2 zh[K], zl[K], zw[K];
    float my, mz;                  // 1.5 * 2^23 * unit of h before the y and z passes
    float whole, frac;             // code = whole + frac + H + L
    float tie;                     // 1/2 - the bound of the code's error
    float g[3][K];                 // the filter and the mapping, for the listed voxels
    float a0h, a0l, a1h, a1l, qmax;
};

// The split weights of the vectors g with the mapping of job J, where make_split_plan accepts them.
template <int K>
bool split_weights(const Job& J, const float* const g[3], SplitW<K>& S)
{
    SplitPlan p;
    if (!make_split_plan(p, K, g, J.sfmt, J.a0, J.a0lo, J.a1, J.a1lo)) return false;
    for (int i = 0; i < K; ++i) {
        S.xh[i] = make_float2(p.hi[0][i], p.hi[0][i]);
        S.xl[i] = make_float2(p.lo[0][i], p.lo[0][i]);
        S.yh[i] = make_float2(p.hi[1][i], p.hi[1][i]);
        S.yl[i] = make_float2(p.lo[1][i], p.lo[1][i]);
        S.yw[i] = make_float2(g[1][i], g[1][i]);
        S.zh[i] = make_float2(p.hi[2][i], p.hi[2][i]);
        S.zl[i] = make_float2(p.lo[2][i], p.lo[2][i]);
        S.zw[i] = make_float2(p.zg[i], p.zg[i]);
        for (int a = 0; a < 3; ++a) S.g[a][i] = g[a][i];
    }
    S.my = p.my;
    S.mz = p.mz;
    S.whole = p.whole;
    S.frac = p.frac;
    S.tie = p.tie;
    S.a0h = J.a0;
    S.a0l = J.a0lo;
    S.a1h = J.a1;
    S.a1l = J.a1lo;
    S.qmax = J.qmax;
    return true;
}

constexpr int SPLIT_LIST = 512;    // listed voxels that are worked off once there are as many,
constexpr int SPLIT_CHECK = 4;     // looked at every so many planes

template <int K>
__host__ __device__ constexpr size_t smem_bytes_split(int sfmt, bool rows = false)
{
    using Geo = Brick<K, TX, CTY>;
    return 128 + static_cast<size_t>(STAGES) * Geo::stage_bytes(sfmt, rows) +
           3 * static_cast<size_t>(Geo::FH) * TX * 2 * sizeof(float) +     // three (h, l) tiles
           (SPLIT_LIST + SPLIT_CHECK * TX * CTY) * sizeof(uint32_t) + 16;  // list, its length
}

// The code of voxel (x, y, z) by the operations of brick_comp, in its order.
template <int K, int SF>
__device__ __noinline__ unsigned dot2_voxel(const void* src, int nx, int ny, int nz, int x, int y,
                                            int z, const SplitW<K>& G)
{
    constexpr int R = (K - 1) / 2;
    float zs = 0.f, zc = 0.f;
#pragma unroll 1
    for (int c = 0; c < K; ++c) {
        const int64_t pl = static_cast<int64_t>(clampi(z + c - R, 0, nz - 1)) * ny;
        float ys = 0.f, yc = 0.f;
#pragma unroll 1
        for (int b = 0; b < K; ++b) {
            const int64_t row = (pl + clampi(y + b - R, 0, ny - 1)) * nx;
            float v[K];
#pragma unroll
            for (int a = 0; a < K; ++a) {
                const int64_t i = row + clampi(x + a - R, 0, nx - 1);
                v[a] = SF == FMT_U16 ? static_cast<float>(__ldg(static_cast<const uint16_t*>(src) + i))
                                     : static_cast<float>(__ldg(static_cast<const unsigned char*>(src) + i));
            }
            float hs, hc;
            dot2_first_exact(G.g[0][0], v[0], hs, hc);
#pragma unroll
            for (int a = 1; a < K; ++a) dot2_exact(G.g[0][a], v[a], hs, hc);
            if (b == 0)
                dot2_first(G.g[1][0], hs, hc, ys, yc);
            else
                dot2_step(G.g[1][b], hs, hc, ys, yc);
        }
        if (c == 0)
            dot2_first(G.g[2][0], ys, yc, zs, zc);
        else
            dot2_step(G.g[2][c], ys, yc, zs, zc);
    }
    return comp_code(zs, zc, G.a0h, G.a0l, G.a1h, G.a1l, G.qmax);
}

// (H, L) -> (h, l): h the multiple of the unit (m = 1.5 * 2^23 units) next to H + L, l the rest
__device__ __forceinline__ void regrid(float2& H, float2& L, float m)
{
    const float2 h = __fadd2_rn(__fadd2_rn(__fadd2_rn(H, L), make_float2(m, m)), make_float2(-m, -m));
    L = __fadd2_rn(__fadd2_rn(H, make_float2(-h.x, -h.y)), L);
    H = h;
}

// The same by a whole warp: the K^2 rows' x passes on its lanes, the y pass of source plane c
// on lane c, the z pass on every lane, with the same operations in the same order.  A short
// list (a brick's last voxels) then takes one load latency instead of K^2.
template <int K, int SF>
__device__ __noinline__ unsigned dot2_voxel_warp(const void* src, int nx, int ny, int nz, int x, int y,
                                                 int z, const SplitW<K>& G)
{
    constexpr int R = (K - 1) / 2, NR = (K * K + 31) / 32;
    const int lane = threadIdx.x & 31;
    float hs[NR], hc[NR];
#pragma unroll
    for (int n = 0; n < NR; ++n) {
        const int e = min(lane + 32 * n, K * K - 1);
        const int c = e / K, b = e - c * K;
        const int64_t row = (static_cast<int64_t>(clampi(z + c - R, 0, nz - 1)) * ny +
                             clampi(y + b - R, 0, ny - 1)) * nx;
        float v[K];
#pragma unroll
        for (int a = 0; a < K; ++a) {
            const int64_t i = row + clampi(x + a - R, 0, nx - 1);
            v[a] = SF == FMT_U16 ? static_cast<float>(__ldg(static_cast<const uint16_t*>(src) + i))
                                 : static_cast<float>(__ldg(static_cast<const unsigned char*>(src) + i));
        }
        dot2_first_exact(G.g[0][0], v[0], hs[n], hc[n]);
#pragma unroll
        for (int a = 1; a < K; ++a) dot2_exact(G.g[0][a], v[a], hs[n], hc[n]);
    }
    float ys = 0.f, yc = 0.f;
    const int c = min(lane, K - 1);
#pragma unroll
    for (int b = 0; b < K; ++b) {
        const int e = c * K + b;
        float s = 0.f, t = 0.f;
#pragma unroll
        for (int n = 0; n < NR; ++n) {
            const float sn = __shfl_sync(0xFFFFFFFFu, hs[n], e & 31), tn = __shfl_sync(0xFFFFFFFFu, hc[n], e & 31);
            if (NR == 1 || (e >> 5) == n) {
                s = sn;
                t = tn;
            }
        }
        if (b == 0)
            dot2_first(G.g[1][0], s, t, ys, yc);
        else
            dot2_step(G.g[1][b], s, t, ys, yc);
    }
    float zs = 0.f, zc = 0.f;
#pragma unroll
    for (int c2 = 0; c2 < K; ++c2) {
        const float s = __shfl_sync(0xFFFFFFFFu, ys, c2), t = __shfl_sync(0xFFFFFFFFu, yc, c2);
        if (c2 == 0)
            dot2_first(G.g[2][0], s, t, zs, zc);
        else
            dot2_step(G.g[2][c2], s, t, zs, zc);
    }
    return comp_code(zs, zc, G.a0h, G.a0l, G.a1h, G.a1l, G.qmax);
}

// ROTZ: as in brick(); the accumulator slots are shifted after each plane, or the plane loop
// is unrolled K times and they rotate at compile time.
template <int K, int SF, class Wt, int LM = LM_ANY, bool ROI = false, bool ROTZ = true, bool BULK = false>
__device__ __forceinline__ bool brick_split(const Job& J, const Wt& G, const CUtensorMap* tmap,
                                            int bx, int by, int bz, unsigned char* smem,
                                            uint32_t& gplane, uint32_t& xphase, unsigned* status)
{
    __builtin_assume(threadIdx.x < NT);   // every launch of a brick has NT threads
    using Geo = Brick<K, TX, CTY>;
    constexpr int R = Geo::R, FH = Geo::FH;
    constexpr int XGROUPS = TX / 4;
    constexpr int XITEMS = FH * XGROUPS;
    constexpr int ES = fmt_bytes(SF), XA = fmt_xalign(SF);

    uint64_t* bars = reinterpret_cast<uint64_t*>(smem);
    const bool tma = LM == LM_TMA || (LM == LM_ANY && J.use_tma);
    const bool rows = LM == LM_ROWS || (LM == LM_ANY && J.rows);
    const int rawb = Geo::stage_bytes(SF, rows);
    const int pitch = rows ? Geo::row_pitch(SF) : Geo::raw_w(SF) * ES;
    constexpr uint32_t txb = Geo::raw_tx(SF);
    unsigned char* raw = smem + 128;
    float* T = reinterpret_cast<float*>(raw + STAGES * rawb);   // tile [plane % 3][h, l][FH][TX]
    uint32_t* list = reinterpret_cast<uint32_t*>(T + 6 * FH * TX);
    volatile uint32_t* count = list + SPLIT_LIST + SPLIT_CHECK * TX * CTY;
    uint64_t* xbar = &bars[XBAR];
    const uint32_t gx = xphase;

    const int tid = threadIdx.x;
    const int tx = tid % BX, ty = tid / BX;
    const int x0 = (ROI ? J.ox0 : 0) + bx * TX, y0 = (ROI ? J.oy0 : 0) + by * CTY;
    const int zc0 = (ROI ? J.oz0 : 0) + bz * J.zchunk;
    const int zc1 = min(zc0 + J.zchunk, ROI ? J.sz1 : J.nz);
    if (zc0 >= zc1) return true;
    const int pfirst = zc0 - R;
    const int nplanes = zc1 - zc0 + 2 * R;
    const uint32_t g0 = gplane;

    if (tid == 0) *count = 0;
    __syncthreads();   // before a voxel is listed
    int issued = 0;
    const uint64_t vol_bytes = static_cast<uint64_t>(J.nx) * J.ny * J.nz * ES;
    if (tma && tid == 0) {
        for (int s = 0; s < STAGES && s < nplanes; ++s, ++issued) {
            if (s == 0 && J.withhold_first) continue;
            const uint32_t q = g0 + s;
            mbar_arrive_expect_tx(&bars[q % STAGES], txb);
            tma_load_3d(raw + (q % STAGES) * rawb, tmap, &bars[q % STAGES], x0 - XA, y0 - R,
                        clampi(pfirst + s, 0, J.nz - 1));
        }
    } else if (rows) {
        for (int s = 0; s < STAGES && s < nplanes; ++s) {
            const uint32_t q = g0 + s;
            copy_rows<Geo, BULK, SF>(raw + (q % STAGES) * rawb, &bars[q % STAGES], J.src, vol_bytes, SF,
                                J.nx, J.ny, J.nz, x0, y0, pfirst + s, tid);
        }
        __syncthreads();   // every thread's expect_tx precedes the single arrival
        if (tid == 0)
            for (int s = 0; s < STAGES && s < nplanes; ++s, ++issued) mbar_arrive(&bars[(g0 + s) % STAGES]);
    }

    // (H, L) of the K output planes in progress; slot K-1-c takes tap c, slot 0 completes
    float2 aH[K][RX / 2], aL[K][RX / 2];
#pragma unroll
    for (int s = 0; s < K; ++s)
#pragma unroll
        for (int x = 0; x < RX / 2; ++x) aH[s][x] = aL[s][x] = make_float2(0.f, 0.f);

    const int ox = x0 + tx * RX;
    const int oy = y0 + ty;
    const int nvalid = (ROI ? J.sx1 : J.nx) - ox;
    const int first = (ROI && J.sx0 > ox) ? J.sx0 - ox : 0;   // leading columns outside the region
    const int yend = ROI ? J.sy1 : J.ny;
    const bool xin = x0 - R >= 0 && x0 + TX - 1 + R <= J.nx - 1;
    // A wait ends by the clock, so one warp may give up a wait that another one sees end.  All lanes
    // of a warp give up together (GONE), and a warp that is gone makes no more arrivals, so no other
    // one gets past the wait for the plane it did not reach: they are gone one limit later at the
    // latest.  Until then it takes part in the CTA's barriers only, of which the votes end the
    // brick for all warps at once (FAILED): one every SPLIT_CHECK planes and one after the last.
    enum { RUNS, GONE, FAILED };
    int state = RUNS;

    // evaluates the listed voxels again (all threads; the caller synchronises around it): a
    // thread per voxel if there are many, a warp per voxel if few
    auto work_off = [&]() {
        const uint32_t n = *count;
        const bool warp = n < NT;
        for (uint32_t i = warp ? tid >> 5 : tid; i < n; i += warp ? NT / 32 : NT) {
            const uint32_t e = list[i];
            const int x = x0 + static_cast<int>(e & (TX - 1));
            const int y = y0 + static_cast<int>((e / TX) & (CTY - 1));
            const int z = zc0 + static_cast<int>(e / (TX * CTY));
            const unsigned code = warp ? dot2_voxel_warp<K, SF>(J.src, J.nx, J.ny, J.nz, x, y, z, G)
                                       : dot2_voxel<K, SF>(J.src, J.nx, J.ny, J.nz, x, y, z, G);
            const int64_t idx = (static_cast<int64_t>(z) * J.ny + y) * J.nx + x;
            if (warp && (tid & 31) != 0) continue;
            if (J.dfmt == FMT_U16)
                static_cast<uint16_t*>(J.dst)[idx] = static_cast<uint16_t>(code);
            else
                static_cast<unsigned char*>(J.dst)[idx] = static_cast<unsigned char>(code);
        }
    };

    // waits for the source plane `it`
    auto loaded = [&](const int it) {
        return !(tma || rows) || mbar_wait(&bars[(g0 + it) % STAGES], ((g0 + it) / STAGES) & 1);
    };

    // The x pass of plane `it` (which is loaded) into tile it % 3.
    auto x_pass = [&](const int it) {
        const uint32_t q = g0 + it;
        const int s = q % STAGES;
        const unsigned char* rs = raw + s * rawb;
        if (!tma && !rows) {
            fill_raw_plain<Geo, NT>(const_cast<unsigned char*>(rs), J.src, SF, J.nx, J.ny, J.nz, x0,
                                    y0, pfirst + it, tid);
            __syncthreads();
        }
        float* Th = T + (it % 3) * 2 * FH * TX;
        float* Tl = Th + FH * TX;
        {
            const uint32_t zterm = static_cast<uint32_t>(clampi(pfirst + it, 0, J.nz - 1)) *
                                   static_cast<uint32_t>(J.ny) * static_cast<uint32_t>(J.nx);
#pragma unroll
            for (int n = 0; n < (XITEMS + NT - 1) / NT; ++n) {
                const int item = tid + n * NT;
                if (item < XITEMS) {
                    const int row = item / XGROUPS, g = item - row * XGROUPS;
                    const int gy = clampi(y0 - R + row, 0, J.ny - 1);
                    const uint32_t sh = rows ? row_shift_elems(zterm, gy, J.nx, x0, XA, SF) : 0u;
                    float win[K + 3];
                    window<K, SF, LM == LM_TMA, true>(rs + (gy - (y0 - R)) * pitch, 4 * g + XA - R, sh,
                                                      win);
                    if (!xin) clamp_window<K>(win, x0 + 4 * g, J.nx);
                    float2 H[2], L[2];
#pragma unroll
                    for (int x = 0; x < 2; ++x)
#pragma unroll
                        for (int a = 0; a < K; ++a) {
                            const float2 v2 = make_float2(win[2 * x + a], win[2 * x + a + 1]);
                            const float2 wh = G.xh[a];
                            const float2 wl = G.xl[a];
                            H[x] = a == 0 ? __fmul2_rn(wh, v2) : __ffma2_rn(wh, v2, H[x]);
                            L[x] = a == 0 ? __fmul2_rn(wl, v2) : __ffma2_rn(wl, v2, L[x]);
                        }
                    regrid(H[0], L[0], G.my);
                    regrid(H[1], L[1], G.my);
                    const float4 oh = make_float4(H[0].x, H[0].y, H[1].x, H[1].y);
                    const float4 ol = make_float4(L[0].x, L[0].y, L[1].x, L[1].y);
                    *reinterpret_cast<float4*>(Th + row * TX + 4 * g) = oh;
                    *reinterpret_cast<float4*>(Tl + row * TX + 4 * g) = ol;
                }
            }
        }
        __syncwarp();
        if ((tid & 31) == 0) mbar_arrive(xbar);
    };

    // Plane `it`: the x pass of the plane after it, then its own y and z passes.  A warp arrives at
    // xbar when its x pass of a plane is written and waits there one plane later, after the y and
    // z passes in between, so the uneven x pass (FH * 16 items on 256 threads) and whatever else
    // delays a warp is waited for only if it lasts longer than those.  With three tiles the wait
    // for plane `it` also says that tile (it + 1) % 3 is free: a warp that has arrived for plane
    // `it` is done with plane it - 2.
    auto plane = [&](const int it, const int u) {
        const uint32_t q = g0 + it;
        const int s = q % STAGES;
        if (!__all_sync(0xFFFFFFFFu, mbar_wait(xbar, (gx + it) & 1) && (it + 1 >= nplanes || loaded(it + 1)))) {
            state = GONE;
            return;
        }
        // stage s is read
        if (rows && tid == 0 && it > 0 && it - 1 + STAGES < nplanes) {
            mbar_arrive(&bars[(q - 1) % STAGES]);   // of the refill before this one
            ++issued;
        }
        if (tma && tid == 0 && it + STAGES < nplanes) {
            mbar_arrive_expect_tx(&bars[s], txb);
            tma_load_3d(raw + s * rawb, tmap, &bars[s], x0 - XA, y0 - R,
                        clampi(pfirst + it + STAGES, 0, J.nz - 1));
            ++issued;
        } else if (rows && it + STAGES < nplanes) {
            // all threads; the arrival follows the next plane's wait
            copy_rows<Geo, BULK, SF>(raw + s * rawb, &bars[s], J.src, vol_bytes, SF, J.nx, J.ny, J.nz, x0,
                                y0, pfirst + it + STAGES, tid);
        }
        if (it % SPLIT_CHECK == SPLIT_CHECK - 1 && __syncthreads_or(*count >= SPLIT_LIST)) {
            if (__syncthreads_or(0)) {   // a warp is gone
                state = FAILED;
                return;
            }
            work_off();
            __syncthreads();
            if (tid == 0) *count = 0;
            __syncthreads();
        }
        if (it + 1 < nplanes) x_pass(it + 1);
        const float* Th = T + (it % 3) * 2 * FH * TX;
        const float* Tl = Th + FH * TX;
        // y pass
        float2 H[RX / 2], L[RX / 2];
#pragma unroll
        for (int b = 0; b < K; ++b) {
            const float4 vh = *reinterpret_cast<const float4*>(Th + (ty + b) * TX + tx * RX);
            const float4 vl = *reinterpret_cast<const float4*>(Tl + (ty + b) * TX + tx * RX);
            const float2 h2[2] = {make_float2(vh.x, vh.y), make_float2(vh.z, vh.w)};
            const float2 l2[2] = {make_float2(vl.x, vl.y), make_float2(vl.z, vl.w)};
            const float2 wh = G.yh[b], wl = G.yl[b];
            const float2 wg = G.yw[b];
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                H[x] = b == 0 ? __fmul2_rn(wh, h2[x]) : __ffma2_rn(wh, h2[x], H[x]);
                L[x] = b == 0 ? __fmul2_rn(wl, h2[x]) : __ffma2_rn(wl, h2[x], L[x]);
                L[x] = __ffma2_rn(wg, l2[x], L[x]);
            }
        }
        // to (h, l) again, then the z pass into the K planes
        regrid(H[0], L[0], G.mz);
        regrid(H[1], L[1], G.mz);
#pragma unroll
        for (int c = 0; c < K; ++c) {
            const int sl = ROTZ ? K - 1 - c : ((u - c + R) % K + K) % K;
            const float2 wh = G.zh[c], wl = G.zl[c];
            const float2 wg = G.zw[c];
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                aH[sl][x] = c == 0 ? __fmul2_rn(wh, H[x]) : __ffma2_rn(wh, H[x], aH[sl][x]);
                aL[sl][x] = c == 0 ? __fmul2_rn(wl, H[x]) : __ffma2_rn(wl, H[x], aL[sl][x]);
                aL[sl][x] = __ffma2_rn(wg, L[x], aL[sl][x]);
            }
        }
        const int sl0 = ROTZ ? 0 : ((u - R) % K + K) % K;
        if (it >= 2 * R && oy < yend && nvalid > 0) {
            const int oz = pfirst + it - R;
            unsigned code[RX];
            float rest[RX];
#pragma unroll
            for (int x = 0; x < RX / 2; ++x) {
                const float2 big = make_float2(12582912.f, 12582912.f), nbig = make_float2(-12582912.f, -12582912.f);
                const float2 Hx = aH[sl0][x];
                const float2 m0 = __fadd2_rn(__fadd2_rn(Hx, big), nbig);         // nearest integer of H
                const float2 s2 = __fadd2_rn(__fadd2_rn(Hx, make_float2(-m0.x, -m0.y)),
                                             __fadd2_rn(aL[sl0][x], make_float2(G.frac, G.frac)));
                const float2 m1 = __fadd2_rn(__fadd2_rn(s2, big), nbig);
                const float2 r = __fadd2_rn(s2, make_float2(-m1.x, -m1.y));      // exact
                const float2 qf = __fadd2_rn(m0, __fadd2_rn(m1, make_float2(G.whole, G.whole)));
                rest[2 * x] = fabsf(r.x);
                rest[2 * x + 1] = fabsf(r.y);
                // an integer in [0, 2^16) added to 2^23 stands in the low bits
                code[2 * x] = __float_as_uint(fminf(fmaxf(qf.x, 0.f), G.qmax) + 8388608.f) & 0xFFFFu;
                code[2 * x + 1] = __float_as_uint(fminf(fmaxf(qf.y, 0.f), G.qmax) + 8388608.f) & 0xFFFFu;
            }
            const bool near_tie = fmaxf(fmaxf(rest[0], rest[1]), fmaxf(rest[2], rest[3])) >= G.tie;
            const int64_t idx = (static_cast<int64_t>(oz) * J.ny + oy) * J.nx + ox;
            store_codes<RX>(J.dst, J.dfmt, idx, first, nvalid, code);
            if (near_tie) {
                const uint32_t at = (static_cast<uint32_t>(oz - zc0) * CTY + ty) * TX + tx * RX;
#pragma unroll
                for (int x = 0; x < RX; ++x)
                    if (rest[x] >= G.tie && x >= first && x < nvalid)
                        list[atomicAdd(const_cast<uint32_t*>(count), 1u)] = at + x;
            }
        }
        if constexpr (ROTZ) {
#pragma unroll
            for (int t = 0; t + 1 < K; ++t)
#pragma unroll
                for (int x = 0; x < RX / 2; ++x) {
                    aH[t][x] = aH[t + 1][x];
                    aL[t][x] = aL[t + 1][x];
                }
        }
    };
    int at = 0;   // the plane a warp is at, or was when it left (-1: before the first)
    if (__all_sync(0xFFFFFFFFu, loaded(0))) {
        x_pass(0);
        if constexpr (ROTZ) {
#pragma unroll 1
            for (; at < nplanes; ++at) {
                plane(at, 0);
                if (state != RUNS) break;
            }
        } else {
#pragma unroll 1
            for (; at < nplanes && state == RUNS; at += K) {
#pragma unroll
                for (int u = 0; u < K; ++u) {
                    if (at + u >= nplanes) break;
                    plane(at + u, u);
                    if (state != RUNS) {
                        at += u - K;
                        break;
                    }
                }
            }
        }
    } else {
        state = GONE;
        at = -1;
    }
    // a warp that is gone: the barriers of the planes it does not take, up to a vote
#pragma unroll 1
    for (int it = max(at, 0); state == GONE && it < nplanes; ++it) {
        if (it % SPLIT_CHECK == SPLIT_CHECK - 1) {
            __syncthreads_or(1);
            __syncthreads_or(1);
            state = FAILED;
        } else if (!tma && !rows && it + 1 < nplanes) {
            __syncthreads();
        }
    }
    if (tma || rows) gplane = g0 + nplanes;
    xphase = gx + nplanes;
    if (!tma) fence_proxy_async();   // a next brick's tensor-map loads may refill these stages
    // the last vote; also, every voxel is listed and its first code stored
    if (state != FAILED && __syncthreads_or(state == GONE)) state = FAILED;
    if (state == FAILED) {
        if (tid == 0) {
            atomicOr(status, STATUS_TIMEOUT);
            // the refills after the planes before `at` and, by other warps that got past their wait
            // for it, after `at`: those whose copies are in flight still need their arrival before
            // the drain
            for (; rows && issued < min(at + STAGES + 1, nplanes); ++issued)
                mbar_arrive(&bars[(g0 + issued) % STAGES]);
            for (int it = issued - 1; it >= 0 && it >= issued - STAGES; --it)
                if (it != 0 || !J.withhold_first)
                    mbar_wait(&bars[(g0 + it) % STAGES], ((g0 + it) / STAGES) & 1);
        }
        __syncthreads();
        return false;
    }
    work_off();
    __syncthreads();   // before a next brick clears the list
    return true;
}

}  // namespace sep
}  // namespace vkt
