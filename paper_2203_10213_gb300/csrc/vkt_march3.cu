// vkt_march3.cu -- dense 3^3 filters of float32 volumes without a shared float tile.
//
// The general direct kernel (vkt_direct.cuh) copies each plane from its stage into a clamped tile
// behind a CTA barrier and reads its windows from there.  A float32 stage needs no conversion: here
// a thread owns 4 columns x 4 rows and walks down the 6 rows they depend on, reading each row's
// window of 6 voxels from the TMA stage and multiplying it into the 3 x 4 x 4 accumulators of the
// output planes and rows it reaches, the x taps of neighbouring outputs as packed FMAs.  No tile and
// no CTA barrier: a stage is refilled once every warp has arrived at its "empty" barrier.  The taps
// are added in the general kernel's order, so the results are the same bits.
// Bound by the FMA pipe (216 packed FMAs of two cycles for 16 voxels, half the time) and HBM traffic:
// 512^3 216 -> 198 us (5.4 TB/s), 256x256x200 28.6 -> 26.2, 208x200x200 28.0 -> 21.6.  Integer sources gain
// nothing (their windows are converted 1.5 times over): 512^3 uint8 -> float32 195 / 189, into uint8
// 226 / 270.
#include <algorithm>
#include <cstdio>
#include <type_traits>

#include "vkt_internal.h"
#include "vkt_tile.cuh"

namespace vkt {
namespace {

constexpr int K = 3, R = 1, XA = 4;
constexpr int NT = 128, RY = 4, TX = 128, TY = (NT / 32) * RY;
constexpr int STAGES = 6;
using Geo = Brick<K, TX, TY>;
constexpr int PITCH = Geo::raw_w(FMT_F32);                 // floats
constexpr int STAGE = Geo::raw_bytes(FMT_F32);
constexpr int SMEM = 128 + STAGES * STAGE;

struct MarchArgs {
    void* dst;
    int nx, ny, nz;
    int zchunk, gzv;            // gzv: z chunks per volume
    int withhold;               // fault injection: arrivals that the first plane's wait lacks
    int64_t vs_dst;             // voxels from one volume's destination to the next
    float w[27];
    float a0, a1, qmax;
    unsigned* status;
};

__global__ void __launch_bounds__(NT, 4)
    k_march3(const __grid_constant__ CUtensorMap tmap, const MarchArgs p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + STAGES;
    unsigned char* raw = smem + 128;
    __builtin_assume(threadIdx.x < NT);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int vol = static_cast<int>(blockIdx.z) / p.gzv;
    const int zc0 = (static_cast<int>(blockIdx.z) - vol * p.gzv) * p.zchunk, zc1 = min(zc0 + p.zchunk, p.nz);
    const int nplanes = zc1 - zc0 + 2 * R, pfirst = zc0 - R;
    float* dst = static_cast<float*>(p.dst) + vol * p.vs_dst;
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
        mbar_arrive_expect_tx(&full[s], Geo::raw_tx(FMT_F32));
        tma_load_4d(raw + s * STAGE, &tmap, &full[s], x0 - XA, y0 - R, clampi(pfirst + it, 0, p.nz - 1), vol);
        ++issued;
    };
    if (tid == 0)
        for (int it = 0; it < STAGES && it < nplanes; ++it) issue(it);

    const int gx = x0 + 4 * lane, gy = y0 + warp * RY;
    const int nvalid = p.nx - gx;
    const bool lface = x0 == 0, rface = x0 + TX - 1 + R > p.nx - 1;   // the tile touches a face
    // rows of the thread's windows, clamped to the volume, as stage offsets of their first voxel
    int off[RY + K - 1];
#pragma unroll
    for (int j = 0; j < RY + K - 1; ++j)
        off[j] = (clampi(gy - R + j, 0, p.ny - 1) - (y0 - R)) * PITCH + 4 * lane + XA - R;

    float2 acc[K][RY][2];
#pragma unroll
    for (int c = 0; c < K; ++c)
#pragma unroll
        for (int i = 0; i < RY; ++i) acc[c][i][0] = acc[c][i][1] = make_float2(0.f, 0.f);
    bool ok = true;        // of the warp
    bool refills = true;   // of thread 0, which loads the stages

    auto plane = [&](const int it, auto uc) {
        constexpr int u = decltype(uc)::value;   // it % K
        const int s = it % STAGES;
        if (!__all_sync(0xFFFFFFFFu, mbar_wait(&full[s], (it / STAGES) & 1))) {   // a warp gives up together
            ok = false;
            return;
        }
        const float* rs = reinterpret_cast<const float*>(raw + s * STAGE);
#pragma unroll
        for (int j = 0; j < RY + K - 1; ++j) {
            const float* q = rs + off[j];
            const float4 m = *reinterpret_cast<const float4*>(q + 1);
            float win[K + 3] = {q[0], m.x, m.y, m.z, m.w, q[5]};
            if (lface) win[0] = lane == 0 ? win[1] : win[0];
            // (rows of whole 16 bytes end with a whole group of four)
            if (rface) win[5] = nvalid == 4 ? win[4] : win[5];
#pragma unroll
            for (int b = 0; b < K; ++b) {
                const int i = j - b;
                if (i < 0 || i >= RY) continue;
#pragma unroll
                for (int c = 0; c < K; ++c) {
                    const int sl = (u + R + 2 * K - c) % K;
#pragma unroll
                    for (int a = 0; a < K; ++a) {
                        const float w = p.w[(c * K + b) * K + a];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const float2 v = make_float2(win[2 * h + a], win[2 * h + a + 1]);
                            float2& d = acc[sl][i][h];
                            d = (c == 0 && b == 0 && a == 0) ? __fmul2_rn(make_float2(w, w), v)
                                                             : __ffma2_rn(make_float2(w, w), v, d);
                        }
                    }
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);   // this warp has read the stage
        constexpr int sl0 = (u - R + K) % K;
        if (it >= 2 * R && nvalid > 0) {
#pragma unroll
            for (int i = 0; i < RY; ++i) {
                const int oy = gy + i;
                if (oy < p.ny) {
                    const int64_t idx = (static_cast<int64_t>(pfirst + it - R) * p.ny + oy) * p.nx + gx;
                    const float v[4] = {acc[sl0][i][0].x, acc[sl0][i][0].y, acc[sl0][i][1].x, acc[sl0][i][1].y};
                    store_row<4>(dst, FMT_F32, idx, nvalid, v, p.a0, p.a1, p.qmax);
                }
            }
        }
        // the stage before this one is free once the slowest warp has read it
        const int refill = it - 1 + STAGES;
        if (tid == 0 && it >= 1 && refill < nplanes) {
            // (a refill that is not made ends every warp's march at the wait for its plane)
            refills = refills && mbar_wait(&empty[refill % STAGES], ((it - 1) / STAGES) & 1);
            if (refills) issue(refill);
        }
        __syncwarp();
    };
#pragma unroll 1
    for (int it = 0; it < nplanes; it += K) {
        plane(it, std::integral_constant<int, 0>{});
        if (!ok || it + 1 >= nplanes) break;
        plane(it + 1, std::integral_constant<int, 1>{});
        if (!ok || it + 2 >= nplanes) break;
        plane(it + 2, std::integral_constant<int, 2>{});
        if (!ok) break;
    }
    if (!ok) atomicOr(p.status, STATUS_TIMEOUT);
    __syncthreads();   // every warp's march has ended
    // every load issued is waited for before the CTA's shared memory is released
    if (tid == 0) {
        if (p.withhold) mbar_arrive(&full[0]);
        for (int it = std::max(0, issued - STAGES); it < issued; ++it) mbar_wait(&full[it % STAGES], (it / STAGES) & 1);
    }
}

}  // namespace

// Launches the march where it serves the job: *taken false otherwise.  Whole float32 volumes (a batch
// of them evenly spaced) that a tensor map describes, into float32 on 16 bytes, at least one tile (128
// columns) wide with three quarters of the tiles' columns in use, and large enough that 128 x 16 tiles in chunks
// of 8 planes give every SM its four CTAs; smaller ones have the one-row shape of the general kernel.
vktError launch_march3(const Job& job, const float* w, const Ctx& ctx, bool* taken)
{
    *taken = false;
    const int nvol = std::max(job.nvol, 1);
    if (job.roi || job.sfmt != FMT_F32 || job.nx < TX) return VKT_NO_ERROR;
    if (store_format(job.dfmt, job.dst, nvol > 1 ? job.vs_dst : 0) != FMT_F32) return VKT_NO_ERROR;
    const int tx = (job.nx + TX - 1) / TX, ty = (job.ny + TY - 1) / TY;
    if (4 * static_cast<long>(job.nx) < 3L * tx * TX) return VKT_NO_ERROR;
    if (static_cast<long>(tx) * ty * (job.nz / 8) * nvol < 4L * ctx.sms) return VKT_NO_ERROR;
    alignas(64) CUtensorMap map;
    if (!encode_tensor_map(&map, FMT_F32, job.src, job.nx, job.ny, job.nz, nvol, job.vs_src, Geo::raw_w(FMT_F32),
                           Geo::FH, 1))
        return VKT_NO_ERROR;
    MarchArgs a;
    a.dst = job.dst;
    a.nx = job.nx;
    a.ny = job.ny;
    a.nz = job.nz;
    a.vs_dst = job.vs_dst;
    for (int i = 0; i < 27; ++i) a.w[i] = w[i];
    a.a0 = job.a0;
    a.a1 = job.a1;
    a.qmax = job.qmax;
    a.withhold = (ctx.debug & VKT_DEBUG_INJECT_WAIT_TIMEOUT) ? 1 : 0;
    a.status = ctx.status;
    int per_sm = 1;
    const vktError ve = prepare_kernel(ctx, reinterpret_cast<const void*>(k_march3), NT, SMEM, &per_sm);
    if (ve != VKT_NO_ERROR) return ve;
    a.zchunk = job.zchunk > 0 ? std::min(job.zchunk, job.nz)
                              : zchunk_direct(static_cast<long>(tx) * ty * nvol, job.nz, ctx.sms, per_sm, R);
    a.gzv = (job.nz + a.zchunk - 1) / a.zchunk;
    if (ty > 65535 || a.gzv > 65535 / nvol) return VKT_NO_ERROR;
    *taken = true;
    if (ctx.debug & VKT_DEBUG_LOG)
        fprintf(stderr, "[vkt] direct-march k=3 grid=(%d,%d,%d) zchunk=%d smem=%d\n", tx, ty, a.gzv * nvol, a.zchunk,
                SMEM);
    const cudaError_t e = launch_pdl(k_march3, dim3(tx, ty, a.gzv * nvol), dim3(NT), SMEM, ctx.stream, map, a);
    count_launches(1);
    if (e != cudaSuccess) return from_cuda(e);
    return from_cuda(cudaGetLastError());
}

}  // namespace vkt
