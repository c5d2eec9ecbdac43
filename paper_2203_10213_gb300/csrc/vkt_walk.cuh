// vkt_walk.cuh -- the separable filter for k = 3 and 5 in registers: every thread computes the x pass
// of the rows it needs itself, straight from the raw stage.
//
// The brick of vkt_sep_brick.cuh shares its x pass through shared memory: a tile written and read per
// plane and a CTA barrier per plane, issue at 60 %.  Here a thread owns 4 columns x RY = 4 rows and
// walks down the RY + k - 1 rows they depend on: the x pass of a row (its window read from the raw
// stage), added into the y sums of the rows it belongs to; the finished y sums go into the k rotating
// z accumulators, one of which is stored per plane.  The x pass is computed 1.5 times over at k = 3 and
// twice at k = 5, but there is no tile and no CTA barrier (a stage is refilled once every warp has
// arrived at its "empty" barrier, so the warps drift apart by up to the stages in flight).  Small CTAs
// (128 threads, 128 x 16 outputs) at three per SM: 512^3 uint8 k = 3 122 us, with 192 threads 139.
// At k = 7 the x pass would be computed 2.5 times and the accumulators alone take 112 registers.
// Every sum is added in the brick's order, so the results are the same bits.  launch_walk_k says
// where it is the faster one; what bounds it is issue (37 instructions per voxel at k = 5 on uint8,
// two conversions of them per voxel) and, for float32 at k = 3, HBM traffic (6.3 TB/s).
#pragma once

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <type_traits>

#include "vkt_internal.h"
#include "vkt_tile.cuh"
#include "vkt_window.cuh"

namespace vkt {
namespace walk {

constexpr int NT = 128, RY = 4, TX = 128, TY = (NT / 32) * RY;
constexpr int STAGES = 6;

template <int K>
struct W {
    float gx[K], gy[K], gz[K];
};

struct Args {
    void* dst;
    int nx, ny, nz;
    int zchunk;
    int withhold;          // fault injection: arrivals that the first plane's wait lacks
    int dfmt;
    float a0, a1, qmax;
    unsigned* status;
};

template <int K, int SF>
struct Cfg {
    using Geo = Brick<K, TX, TY>;
    static constexpr int ES = fmt_bytes(SF);
    static constexpr int PITCH = Geo::raw_w(SF) * ES;
    static constexpr int STAGE = Geo::raw_bytes(SF);
    static constexpr int SMEM = 128 + STAGES * STAGE;
    static_assert(2 * STAGES * 8 <= 128, "barriers in the header");
};

template <int K, int SF, bool OUT_F32>
__global__ void __launch_bounds__(NT, 3)
    k_walk(const __grid_constant__ CUtensorMap tmap, const Args p, const W<K> G)
{
    using C = Cfg<K, SF>;
    using Geo = typename C::Geo;
    constexpr int R = Geo::R, XA = fmt_xalign(SF), NW = K + 3;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + STAGES;
    unsigned char* raw = smem + 128;
    __builtin_assume(threadIdx.x < NT);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int zc0 = blockIdx.z * p.zchunk, zc1 = min(zc0 + p.zchunk, p.nz);
    const int nplanes = zc1 - zc0 + 2 * R, pfirst = zc0 - R;
    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], s == 0 ? 1 + p.withhold : 1);
            mbar_init(&empty[s], NT / 32);
        }
        fence_mbar_init();
        prefetch_tensor_map(&tmap);
    }
    __syncthreads();
    grid_dependency_wait();   // programmatic launch: the previous kernel's writes are visible
    launch_dependents();
    int issued = 0;
    auto issue = [&](int it) {
        const int s = it % STAGES;
        mbar_arrive_expect_tx(&full[s], Geo::raw_tx(SF));
        tma_load_3d(raw + s * C::STAGE, &tmap, &full[s], x0 - XA, y0 - R, clampi(pfirst + it, 0, p.nz - 1));
        ++issued;
    };
    if (tid == 0)
        for (int it = 0; it < STAGES && it < nplanes; ++it) issue(it);

    const int gx = x0 + 4 * lane, gy = y0 + warp * RY;
    const int nvalid = p.nx - gx;
    const bool lface = x0 == 0, rface = x0 + TX - 1 + R > p.nx - 1;   // the tile touches a face
    // rows of the thread's windows, clamped to the volume, as stage offsets of their first columns
    int off[RY + K - 1];
#pragma unroll
    for (int j = 0; j < RY + K - 1; ++j) 
        off[j] = (clampi(gy - R + j, 0, p.ny - 1) - (y0 - R)) * C::PITCH + 4 * lane * C::ES;

    float2 acc[K][RY][2];   // z accumulators
#pragma unroll
    for (int c = 0; c < K; ++c)
#pragma unroll
        for (int i = 0; i < RY; ++i) acc[c][i][0] = acc[c][i][1] = make_float2(0.f, 0.f);
    bool ok = true;        // of the warp
    bool refills = true;   // of thread 0, which loads the stages

    float2 ysum[RY][2];
    // the x and y passes of plane `it`
    auto xy_pass = [&](const int it) {
        const int s = it % STAGES;
        if (!__all_sync(0xFFFFFFFFu, mbar_wait(&full[s], (it / STAGES) & 1))) {   // a warp gives up together
            ok = false;
            return;
        }
        const unsigned char* rs = raw + s * C::STAGE;
#pragma unroll
        for (int j = 0; j < RY + K - 1; ++j) {
            const unsigned char* row = rs + off[j];
            float win[NW];
            if constexpr (SF == FMT_F32) {
                const float* q = reinterpret_cast<const float*>(row) + XA - R;
                if constexpr (K == 5) {
                    const float2 a = *reinterpret_cast<const float2*>(q);
                    const float4 b = *reinterpret_cast<const float4*>(q + 2);
                    const float2 d = *reinterpret_cast<const float2*>(q + 6);
                    win[0] = a.x; win[1] = a.y; win[2] = b.x; win[3] = b.y;
                    win[4] = b.z; win[5] = b.w; win[6] = d.x; win[7] = d.y;
                } else {
                    const float4 b = *reinterpret_cast<const float4*>(q + 1);
                    win[0] = q[0]; win[1] = b.x; win[2] = b.y; win[3] = b.z; win[4] = b.w; win[5] = q[5];
                }
            } else {
                window<K, SF, true, false>(row, XA - R, 0u, win);
            }
            if (lface) {
#pragma unroll
                for (int e = 0; e < R; ++e) win[e] = lane == 0 ? win[R] : win[e];
            }
            if (rface) {
                // rows of whole 16 bytes end with a whole group of four
#pragma unroll
                for (int e = R + 4; e < NW; ++e) win[e] = nvalid == 4 ? win[R + 3] : win[e];
            }
            // even taps as packed FMAs over neighbouring outputs, whose operand pairs stand side by side;
            // odd taps as single ones (their pairs would have to be moved together first)
            float2 t[2];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int a = 0; a < K; ++a) {
                    const float g = G.gx[a];
                    const float v0 = win[2 * h + a], v1 = win[2 * h + a + 1];
                    if (a == 0) {
                        t[h] = __ffma2_rn(make_float2(g, g), make_float2(v0, v1), make_float2(0.f, 0.f));
                    } else if (a % 2 == 0) {
                        t[h] = __ffma2_rn(make_float2(g, g), make_float2(v0, v1), t[h]);
                    } else {
                        t[h].x = __fmaf_rn(g, v0, t[h].x);
                        t[h].y = __fmaf_rn(g, v1, t[h].y);
                    }
                }
#pragma unroll
            for (int i = 0; i < RY; ++i) {
                const int b = j - i;
                if (b < 0 || b >= K) continue;
                const float2 g = make_float2(G.gy[b], G.gy[b]);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    ysum[i][h] = b == 0 ? __fmul2_rn(g, t[h]) : __ffma2_rn(g, t[h], ysum[i][h]);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);   // this warp has read the stage
        // the stage before this one is free once the slowest warp has read it
        const int refill = it - 1 + STAGES;
        if (tid == 0 && it >= 1 && refill < nplanes) {
            // (a refill that is not made ends every warp's march at the wait for its plane)
            refills = refills && mbar_wait(&empty[refill % STAGES], ((it - 1) / STAGES) & 1);
            if (refills) issue(refill);
        }
        __syncwarp();
    };
    // its z pass, u = it % K: the accumulators rotate at compile time, so this (short) part of a
    // plane's code stands K times; all of it K times overflowed the instruction cache
    auto z_pass = [&](const int it, auto uc) {
        constexpr int u = decltype(uc)::value;
        // slot of the output plane that this plane reaches through tap c
#pragma unroll
        for (int c = 0; c < K; ++c) {
            const int sl = ((u - c + R) % K + K) % K;
            const float2 g = make_float2(G.gz[c], G.gz[c]);
#pragma unroll
            for (int i = 0; i < RY; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    acc[sl][i][h] = c == 0 ? __fmul2_rn(g, ysum[i][h]) : __ffma2_rn(g, ysum[i][h], acc[sl][i][h]);
        }
        const int sl0 = ((u - R) % K + K) % K;
        if (it >= 2 * R && nvalid > 0) {
#pragma unroll
            for (int i = 0; i < RY; ++i) {
                const int oy = gy + i;
                if (oy < p.ny) {
                    const int64_t idx = (static_cast<int64_t>(pfirst + it - R) * p.ny + oy) * p.nx + gx;
                    const float v[4] = {acc[sl0][i][0].x, acc[sl0][i][0].y, acc[sl0][i][1].x, acc[sl0][i][1].y};
                    store_row<4>(p.dst, OUT_F32 ? FMT_F32 : p.dfmt, idx, nvalid, v, p.a0, p.a1, p.qmax);
                }
            }
        }
    };
    int u = 0;
#pragma unroll 1
    for (int it = 0; it < nplanes; ++it) {
        xy_pass(it);
        if (!ok) break;
        switch (u) {
        case 0: z_pass(it, std::integral_constant<int, 0>{}); break;
        case 1: z_pass(it, std::integral_constant<int, 1>{}); break;
        case 2: z_pass(it, std::integral_constant<int, 2>{}); break;
        case 3: if constexpr (K > 3) z_pass(it, std::integral_constant<int, 3 % K>{}); break;
        default: if constexpr (K > 3) z_pass(it, std::integral_constant<int, 4 % K>{}); break;
        }
        u = u + 1 == K ? 0 : u + 1;
    }
    if (!ok) atomicOr(p.status, STATUS_TIMEOUT);
    __syncthreads();   // every warp's march has ended
    // every load issued is waited for before the CTA's shared memory is released
    if (tid == 0) {
        if (p.withhold) mbar_arrive(&full[0]);
        for (int it = std::max(0, issued - STAGES); it < issued; ++it) mbar_wait(&full[it % STAGES], (it / STAGES) & 1);
    }
}

}  // namespace walk

// Launches the walk where it serves the job: *taken false otherwise.  Whole volumes that a tensor map
// describes, one at a time, whose codes FP32 decides, and where it is the faster of the two
// (us, brick / walk):
//   float32 sources wider than 32 columns: 512^3 k = 3 173 / 171, k = 5 254 / 175; 64x300x200 13.3 / 11.6 and
//     23.8 / 16.6; 32x300x100 7.9 / 9.4 and 13.5 / 13.3 (its tile is 128 columns, the brick's 64);
//   integer sources at k = 3, if its tiles cover no more columns than the brick's and give every SM
//     work: uint8 -> float32 512^3 152 / 122, 256x256x200 19.2 / 16.8, 192x200x200 13.3 / 13.6, 128x200x200
//     9.8 / 12.2.  (k = 5: 189 / 189 and into uint8 232 / 249.)
// Sources without a tensor map lose: the shift of every row is worked out k times over.
template <int K>
vktError launch_walk_k(const Job& job, const float* gx, const float* gy, const float* gz, const Ctx& ctx,
                       bool* taken)
{
    using namespace walk;
    using Geo = Brick<K, TX, TY>;
    *taken = false;
    if (job.roi || job.comp || job.nvol > 1) return VKT_NO_ERROR;
    const int tx = (job.nx + TX - 1) / TX, ty = (job.ny + TY - 1) / TY;
    if (job.sfmt == FMT_F32) {
        if (job.nx <= 32 || job.dfmt != FMT_F32) return VKT_NO_ERROR;   // (into codes: compensated)
    } else {
        const int bricks = (job.nx + 63) / 64;
        if (K != 3 || 2 * tx > bricks) return VKT_NO_ERROR;
        if (static_cast<long>(tx) * ty * (job.nz / 8) < 4L * ctx.sms) return VKT_NO_ERROR;
    }
    void (*kern)(const CUtensorMap, const Args, const W<K>) = nullptr;
    size_t smem = 0;
    auto pick = [&](auto sf) {
        constexpr int SF = decltype(sf)::value;
        kern = store_format(job.dfmt, job.dst) == FMT_F32 ? k_walk<K, SF, true> : k_walk<K, SF, false>;
        smem = Cfg<K, SF>::SMEM;
    };
    if (job.sfmt == FMT_F32) pick(std::integral_constant<int, FMT_F32>{});
    if constexpr (K == 3) {
        if (job.sfmt == FMT_U8) pick(std::integral_constant<int, FMT_U8>{});
        if (job.sfmt == FMT_U16) pick(std::integral_constant<int, FMT_U16>{});
    }
    alignas(64) CUtensorMap map;
    if (!encode_tensor_map_3d(&map, job.sfmt, job.src, job.nx, job.ny, job.nz, Geo::raw_w(job.sfmt), Geo::FH, 1))
        return VKT_NO_ERROR;
    Args a;
    a.dst = job.dst;
    a.nx = job.nx;
    a.ny = job.ny;
    a.nz = job.nz;
    a.dfmt = store_format(job.dfmt, job.dst);
    a.a0 = job.a0;
    a.a1 = job.a1;
    a.qmax = job.qmax;
    a.withhold = (ctx.debug & VKT_DEBUG_INJECT_WAIT_TIMEOUT) ? 1 : 0;
    a.status = ctx.status;
    W<K> G;
    for (int i = 0; i < K; ++i) {
        G.gx[i] = gx[i];
        G.gy[i] = gy[i];
        G.gz[i] = gz[i];
    }
    int per_sm = 1;
    const vktError ve = prepare_kernel(ctx, reinterpret_cast<const void*>(kern), NT, smem, &per_sm);
    if (ve != VKT_NO_ERROR) return ve;
    a.zchunk = job.zchunk > 0 ? std::min(job.zchunk, job.nz)
                              : zchunk_direct(static_cast<long>(tx) * ty, job.nz, ctx.sms, per_sm, Geo::R);
    const int tz = (job.nz + a.zchunk - 1) / a.zchunk;
    if (ty > 65535 || tz > 65535) return VKT_NO_ERROR;
    *taken = true;
    if (ctx.debug & VKT_DEBUG_LOG)
        fprintf(stderr, "[vkt] separable-walk k=%d grid=(%d,%d,%d) zchunk=%d smem=%zu\n", K, tx, ty, tz, a.zchunk, smem);
    const cudaError_t e = launch_pdl(kern, dim3(tx, ty, tz), dim3(NT), smem, ctx.stream, map, a, G);
    count_launches(1);
    if (e != cudaSuccess) return from_cuda(e);
    return from_cuda(cudaGetLastError());
}

}  // namespace vkt
