// vkt_star.cu -- dense 3^3 filters whose only taps lie on the axes (the 7-point Laplacian, gradients,
// unsharp masks) on integer volumes: the direct path's result at the price of memory traffic.
//
// The general k = 3 kernel multiplies all 27 taps and is bound by instruction issue (37 per
// voxel).  Here the 20 zero taps are left out (a product with 0 adds nothing to an integer
// source's sum), which also leaves nothing to share between threads but the raw codes: a thread
// reads its 4 x 4 voxels of a plane and their neighbours from the TMA stage as words, keeps the
// plane before in registers, and no converted tile and no CTA barrier are needed.  A warp takes
// 128 columns x 4 rows, a CTA 128 x 32, marching through z; a stage is refilled once every warp
// has arrived at its "empty" barrier.
// The taps are added in the order of the general kernel, (z-1) (y-1) (x-1) (0) (x+1) (y+1) (z+1), so the
// float32 sums are the same.  Bound by HBM traffic: 512^3 uint8 -> float32 194 -> 108 us (6.2 TB/s of
// the 6.8 a copy reaches), into uint8 codes 1637 (Dot2) -> 181 us.
#include <algorithm>
#include <cstdio>

#include "vkt_internal.h"
#include "vkt_list_plan.h"
#include "vkt_tile.cuh"
#include "vkt_window.cuh"

namespace vkt {
namespace {

constexpr int NT = 256, RY = 4, TX = 128, TY = (NT / 32) * RY;
constexpr int STAGES = 8;

// what is stored: float32 values, codes rounded from the FP32 sum, or codes whose sums are exact
// (ListPlan::exact)
enum : int { OUT_F32 = 0, OUT_FP32_CODE = 1, OUT_EXACT_CODE = 2 };

struct StarArgs {
    void* dst;
    int nx, ny, nz;
    int zchunk;
    int withhold;                      // fault injection: arrivals that the first plane's wait lacks
    int dfmt;
    float zm, ym, xm, c, xp, yp, zp;   // the taps
    float a0, a1, qmax;
    float whole, frac;                 // exact codes: whole + frac + sum
    unsigned* status;
};

template <int SF>
struct StarGeo {
    static constexpr int ES = fmt_bytes(SF), XA = fmt_xalign(SF);
    static constexpr int PITCH = TX * ES + 32;          // raw row: 16 bytes on either side
    static constexpr int ROWS = TY + 2;
    static constexpr int STAGE = (PITCH * ROWS + 127) & ~127;
    static constexpr int SMEM = 256 + STAGES * STAGE;
};

template <int SF, int OUT>
__global__ void __launch_bounds__(NT, 2)
    k_star(const __grid_constant__ CUtensorMap tmap, const StarArgs p)
{
    using G = StarGeo<SF>;
    constexpr bool CENTRE = OUT == OUT_EXACT_CODE;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + STAGES;
    unsigned char* raw = smem + 256;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int zc0 = blockIdx.z * p.zchunk, zc1 = min(zc0 + p.zchunk, p.nz);
    const int nplanes = zc1 - zc0 + 2;
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
        mbar_arrive_expect_tx(&full[s], G::PITCH * G::ROWS);
        tma_load_3d(raw + s * G::STAGE, &tmap, &full[s], x0 - G::XA, y0 - 1, clampi(zc0 - 1 + it, 0, p.nz - 1));
        ++issued;
    };
    if (tid == 0)
        for (int it = 0; it < STAGES && it < nplanes; ++it) issue(it);

    const int gx = x0 + 4 * lane, gy = y0 + warp * RY;
    // stage offset of the thread's voxels in rows gy - 1 .. gy + 4, clamped to the volume
    int off[RY + 2];
#pragma unroll
    for (int j = 0; j < RY + 2; ++j)
        off[j] = (clampi(gy - 1 + j, 0, p.ny - 1) - (y0 - 1)) * G::PITCH + (4 * lane + G::XA) * G::ES;
    const bool lface = gx == 0, rface = gx + 4 >= p.nx;

    // voxels 4 lane .. + 3 of a row as pairs, and one voxel
    auto load4 = [&](const unsigned char* q, float2 (&v)[2]) {
        uint32_t w[G::ES];
        if constexpr (SF == FMT_U8) {
            w[0] = *reinterpret_cast<const uint32_t*>(q);
        } else {
            const uint2 t = *reinterpret_cast<const uint2*>(q);
            w[0] = t.x;
            w[1] = t.y;
        }
        v[0] = code_pair<SF, CENTRE>(w, 0);
        v[1] = code_pair<SF, CENTRE>(w, 2);
    };
    auto load1 = [&](const unsigned char* q) {
        const uint32_t c = SF == FMT_U8 ? *q : *reinterpret_cast<const uint16_t*>(q);
        return __uint_as_float(c | 0x4B000000u) -
               (CENTRE ? 8388608.f + (SF == FMT_U8 ? 128.f : 32768.f) : 8388608.f);
    };
    auto two = [](float w) { return make_float2(w, w); };

    float2 acc[RY][2], before[RY][2];   // the sums of plane it - 1, its voxels
#pragma unroll
    for (int i = 0; i < RY; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) acc[i][h] = before[i][h] = make_float2(0.f, 0.f);
    bool ok = true;
#pragma unroll 1
    for (int it = 0; it < nplanes; ++it) {
        const int s = it % STAGES;
        if (!__all_sync(0xFFFFFFFFu, mbar_wait(&full[s], (it / STAGES) & 1))) {   // a warp gives up together
            ok = false;
            break;
        }
        const unsigned char* rs = raw + s * G::STAGE;
        // rows of the plane: the one before, this and the next of a walk down the thread's rows
        float2 up[2], cur[2], down[2];
        load4(rs + off[0], up);
        load4(rs + off[1], cur);
#pragma unroll
        for (int i = 0; i < RY; ++i) {
            load4(rs + off[i + 2], down);
            float left = load1(rs + off[i + 1] - G::ES), right = load1(rs + off[i + 1] + 4 * G::ES);
            left = lface ? cur[0].x : left;
            right = rface ? cur[1].y : right;
            // plane it - 1 takes its last tap and is stored
            float v[4];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 d = __ffma2_rn(two(p.zp), cur[h], acc[i][h]);
                v[2 * h] = d.x;
                v[2 * h + 1] = d.y;
            }
            const int oy = gy + i;
            if (it >= 2 && oy < p.ny && gx < p.nx) {
                const int64_t idx = (static_cast<int64_t>(zc0 + it - 2) * p.ny + oy) * p.nx + gx;
                if constexpr (OUT == OUT_F32) {
                    *reinterpret_cast<float4*>(static_cast<float*>(p.dst) + idx) =
                        make_float4(fmaf(p.a1, v[0], p.a0), fmaf(p.a1, v[1], p.a0), fmaf(p.a1, v[2], p.a0),
                                    fmaf(p.a1, v[3], p.a0));
                } else if constexpr (OUT == OUT_FP32_CODE) {
                    store_row<4>(p.dst, p.dfmt, idx, 4, v, p.a0, p.a1, p.qmax);
                } else {
                    unsigned code[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float m0 = __fsub_rn(__fadd_rn(v[e], 12582912.f), 12582912.f);
                        const float s2 = __fadd_rn(__fsub_rn(v[e], m0), p.frac);
                        const float m1 = __fsub_rn(__fadd_rn(s2, 12582912.f), 12582912.f);
                        const float r = __fsub_rn(s2, m1);
                        float qf = __fadd_rn(m0, __fadd_rn(m1, p.whole));
                        // a tie goes to the even code (the last bit of the integer 1.5 * 2^23 + qf)
                        if (fabsf(r) == 0.5f && (__float_as_uint(__fadd_rn(qf, 12582912.f)) & 1u))
                            qf = __fadd_rn(qf, r > 0.f ? 1.f : -1.f);
                        code[e] = __float_as_uint(fminf(fmaxf(qf, 0.f), p.qmax) + 8388608.f) & 0xFFFFu;
                    }
                    store_codes<4>(p.dst, p.dfmt, idx, 0, 4, code);
                }
            }
            // plane `it` takes all taps but its last
            const float2 lm[2] = {make_float2(left, cur[0].x), make_float2(cur[0].y, cur[1].x)};
            const float2 lp[2] = {lm[1], make_float2(cur[1].y, right)};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float2 d = __fmul2_rn(two(p.zm), before[i][h]);
                d = __ffma2_rn(two(p.ym), up[h], d);
                d = __ffma2_rn(two(p.xm), lm[h], d);
                d = __ffma2_rn(two(p.c), cur[h], d);
                d = __ffma2_rn(two(p.xp), lp[h], d);
                acc[i][h] = __ffma2_rn(two(p.yp), down[h], d);
                before[i][h] = cur[h];
                up[h] = cur[h];
                cur[h] = down[h];
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);
        // the plane before this one: its stage is free once the slowest warp has read it
        const int refill = it - 1 + STAGES;
        if (tid == 0 && it >= 1 && refill < nplanes) {
            // (a refill that is not made ends every warp's march at the wait for its plane)
            if (ok && mbar_wait(&empty[refill % STAGES], ((it - 1) / STAGES) & 1))
                issue(refill);
            else
                ok = false;
        }
        __syncwarp();
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

// Whether the job is a 3^3 filter with taps on the axes only, over one whole integer volume into an
// aligned destination whose codes FP32 decides, or exact sums with the weights of `plan` (job.comp).
// launch_star then asks for a tensor map of the volume.
static bool star_job(const Job& job, const float* w, const Ctx& ctx, ListPlan& plan)
{
    if (job.roi || job.nvol > 1 || job.sfmt == FMT_F32) return false;
    for (int c = 0; c < 3; ++c)
        for (int b = 0; b < 3; ++b)
            for (int a = 0; a < 3; ++a)
                if ((c != 1) + (b != 1) + (a != 1) > 1 && w[(c * 3 + b) * 3 + a] != 0.f) return false;
    for (int i = 0; i < 27; ++i)
        if (!(w[i] - w[i] == 0.f)) return false;   // infinities and NaN take all 27 products
    if (reinterpret_cast<uintptr_t>(job.dst) % 16 != 0) return false;
    if (job.comp)
        return make_list_plan(plan, 3, w, job.sfmt, job.a0, job.a0lo, job.a1, job.a1lo) && plan.exact;
    return true;
}

vktError launch_star(const Job& job, const float* w, const Ctx& ctx, bool* taken)
{
    *taken = false;
    ListPlan plan;
    if (!star_job(job, w, ctx, plan)) return VKT_NO_ERROR;
    const bool u8 = job.sfmt == FMT_U8;
    alignas(64) CUtensorMap map;
    if (!encode_tensor_map_3d(&map, job.sfmt, job.src, job.nx, job.ny, job.nz, TX + 2 * fmt_xalign(job.sfmt),
                              TY + 2, 1))
        return VKT_NO_ERROR;
    *taken = true;
    StarArgs a;
    a.dst = job.dst;
    a.nx = job.nx;
    a.ny = job.ny;
    a.nz = job.nz;
    a.dfmt = job.dfmt;
    const float* t = job.comp ? plan.w : w;
    a.zm = t[4];
    a.ym = t[10];
    a.xm = t[12];
    a.c = t[13];
    a.xp = t[14];
    a.yp = t[16];
    a.zp = t[22];
    a.a0 = job.a0;
    a.a1 = job.a1;
    a.qmax = job.qmax;
    a.whole = job.comp ? plan.whole : 0.f;
    a.frac = job.comp ? plan.frac : 0.f;
    a.withhold = (ctx.debug & VKT_DEBUG_INJECT_WAIT_TIMEOUT) ? 1 : 0;
    a.status = ctx.status;
    const int out = job.dfmt == FMT_F32 ? OUT_F32 : job.comp ? OUT_EXACT_CODE : OUT_FP32_CODE;
    auto kern = u8 ? (out == OUT_F32 ? k_star<FMT_U8, OUT_F32>
                      : out == OUT_FP32_CODE ? k_star<FMT_U8, OUT_FP32_CODE> : k_star<FMT_U8, OUT_EXACT_CODE>)
                   : (out == OUT_F32 ? k_star<FMT_U16, OUT_F32>
                      : out == OUT_FP32_CODE ? k_star<FMT_U16, OUT_FP32_CODE> : k_star<FMT_U16, OUT_EXACT_CODE>);
    const size_t smem = u8 ? StarGeo<FMT_U8>::SMEM : StarGeo<FMT_U16>::SMEM;
    int per_sm = 1;
    const vktError ve = prepare_kernel(ctx, reinterpret_cast<const void*>(kern), NT, smem, &per_sm);
    if (ve != VKT_NO_ERROR) return ve;
    const int gx = (job.nx + TX - 1) / TX, gy = (job.ny + TY - 1) / TY;
    a.zchunk = job.zchunk > 0 ? std::min(job.zchunk, job.nz)
                              : zchunk_direct(static_cast<long>(gx) * gy, job.nz, ctx.sms, per_sm, 1);
    const int gz = (job.nz + a.zchunk - 1) / a.zchunk;
    if (gy > 65535 || gz > 65535) {
        *taken = false;
        return VKT_NO_ERROR;
    }
    if (ctx.debug & VKT_DEBUG_LOG)
        fprintf(stderr, "[vkt] direct-star k=3 grid=(%d,%d,%d) zchunk=%d smem=%zu\n", gx, gy, gz, a.zchunk, smem);
    const cudaError_t e = launch_pdl(kern, dim3(gx, gy, gz), dim3(NT), smem, ctx.stream, map, a);
    count_launches(1);
    if (e != cudaSuccess) return from_cuda(e);
    return from_cuda(cudaGetLastError());
}

}  // namespace vkt
