// vkt_tc.cu -- ApplyFilter on the tcgen05 tensor cores for dense k^3 filters (k = 5, 7, 9)
// on float32 volumes, with a split FP16 hi/lo operand scheme that keeps the result within
// the FP32 path's accuracy.
//
// Formulation.  Fix one input plane z' and one kernel row offset b (dy = b - r).  For the
// 8 outputs x_o of an x tile, the x taps of every kernel plane c are a banded Toeplitz
// product over a 16-wide input window:
//     D[m, (c, j)] += sum_kk  A_b[m, kk] * T_b[kk, (c, j)]
//     A_b[m, kk]   = v(x0 - 4 + 8t + kk, y0 + m + dy, z')          (input rows shifted by dy)
//     T_b[kk,(c,j)] = w[c][b][kk - j - 4 + r]   (zero outside the band)
// so one 128 x N x 16 MMA (M = 128 output rows, N = 8 * slots, slots >= k) yields the
// contribution of plane z' to the k output planes z' - c + r at once.  Summing over b and
// over the three split products A_hi T_hi + A_hi T_lo + A_lo T_hi (each operand split as
// hi = fp16(x s), lo = fp16(x s - hi), s a power of two) happens in the TMEM accumulator;
// the epilogue scales back and adds the k slot columns into k rotating register
// accumulators, one of which completes per input plane (z-march).
//
// The items of a launch may span nvol volumes of equal dims (a training batch): one 128^3 volume
// has too few of them to give every SM one, eight have.
//
// Warp roles (640 threads, one CTA per SM, persistent over (x, y, z-chunk) work items):
//   warp 1         lane 0 issues the MMAs and commits
//   warp 5         lane 0 issues TMA loads of f32 plane tiles
//   warps 4g+0, 2, 3 (g < 3)   convert plane tiles to fp16 hi/lo operands (clamp-to-edge, scale)
//   warps 12..19   epilogue: TMEM -> registers, z-march accumulate, store
// What bounds it: an MMA of 128 x 64 x 16 reads 6 KB of shared memory, 48 of its 53 cycles, one of
// 128 x 128 x 16 8 KB in 69; at k = 7 the 28 MMAs of an item's plane take 1710 of its 2420 cycles, the
// rest is the hand-off between planes and the converters' share of shared memory.  What kept the MMAs
// from that rate, with 1024 x 1024 x 256 at k = 5 / 7 / 9 1413 / 1655 / 2063 us and 128^3 at k = 7 68:
// (1) Warps 1, 5, 9, ... share a scheduler: with converters among them an MMA took 70 to 80 cycles to
// issue.  (2) A converter's loads and stores wait for shared memory behind the MMAs, a plane takes a
// group 5800 cycles, so two operand buffers (and one group) ran dry; hence three groups with a buffer
// each, and the registers moved from them to the epilogue (setmaxnreg).  Both: 1087 / 1413 / 1752, 33.
// (3) STACK below: 967 / 1146, 28.5.
// No gain from: A operands on whole 128-byte lines, collector reuse of A, issuing by the whole warp.
// Every wait is bounded; on a timeout the CTA records it, drains what it issued and exits.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstdio>

#include "vkt_internal.h"
#include "vkt_tile.cuh"

namespace vkt {
namespace {

constexpr int MROWS = 128;                 // output rows per tile (MMA M)
constexpr int XT = 2;                      // x tiles of 8 outputs per work item
constexpr int NCH = XT + 1;                // 8-wide input chunks per plane tile
constexpr int STAGES = 5;
constexpr int CGRP = 3;                    // converter groups, one per operand buffer
constexpr int CONV_WARPS = NCH, NCONV = CONV_WARPS * 32;   // of a group: a warp per chunk
constexpr int MMA_WARP = 1, TMA_WARP = 5, EPI_WARP0 = 12, NEPI = 256;
constexpr int NTHREADS = EPI_WARP0 * 32 + NEPI;
static_assert(CONV_WARPS == 3 && EPI_WARP0 == 4 * CGRP, "three of every four warps convert");
// Registers of a thread at launch, then of the first three warpgroups and of the epilogue's two
// (k = 7 80 and 120: 1417 us, 72 and 128: 1514, where the converters spill, 88 and 104: 1413).
constexpr int REGS = 96, REGS_CONV = 88, REGS_EPI = 104;
static_assert(3 * REGS_CONV + 2 * REGS_EPI <= 5 * REGS && NTHREADS == 5 * 128, "shares of the launch's registers");
constexpr int SC_RING = 8;

template <int K>
struct TcCfg {
    static constexpr int R = (K - 1) / 2;
    static constexpr int ROWS = MROWS + 2 * R;            // input rows of a plane tile
    static constexpr int SLOTS = ((K + 1) / 2) * 2;       // even, so N is a multiple of 16
    static constexpr int N = SLOTS * 8;
    // STACK: A_hi T_hi and A_hi T_lo are one MMA over the stacked operand [T_hi | T_lo] of 2N columns;
    // D's columns [0, N) then hold the hi hi and lo hi products and [N, 2N) the hi lo ones.  An MMA's
    // time is that of its shared memory reads below N = 128 (53 cycles at 64, 69 at 128), so a row
    // offset takes 122 cycles instead of 160.  At k = 9 two buffers of 2N columns do not fit TMEM.
    static constexpr bool STACK = K <= 7;
    static constexpr int DN = STACK ? 2 * N : N;         // TMEM columns per (buffer, x tile)
    static constexpr int DBUF = STACK ? 2 : 3;           // TMEM accumulator buffers
    static_assert(STACK || DBUF == CGRP, "d_full stands in for op_empty");
    static_assert(DBUF * XT * DN <= 512, "TMEM holds 512 columns");
    static constexpr int TMEM_COLS = (DBUF * XT * DN <= 256) ? 256 : 512;
    static constexpr int STAGE_BYTES = ((ROWS * NCH * 8 * 4) + 1023) & ~1023;
    static constexpr int STAGE_TX = ROWS * NCH * 8 * 4;
    // an operand plane: per 8-wide chunk, ROWS rows of 16 bytes (an A operand shifted down by b rows
    // starts 16 b bytes further on)
    static constexpr int CHUNK_BYTES = ROWS * 16;
    static constexpr int OP_BYTES = (NCH * CHUNK_BYTES + 1023) & ~1023;   // one fp16 plane
    static constexpr int B_BYTES = 2 * N * 16;                            // one Toeplitz (hi or lo)
    // converter items of 4 values of a chunk: (row, half) for the first 128 rows, then the last 2R rows
    static constexpr int MAIN = MROWS * 2 / 32;           // items per lane
    static constexpr int EXTRA = 2 * R * 2;               // lanes with one more
    static_assert(EXTRA <= 32, "items of a lane");
    // shared memory map
    static constexpr int OFF_STAGE = 1024;
    static constexpr int OFF_OP = OFF_STAGE + STAGES * STAGE_BYTES;       // [CGRP][hi,lo]
    static constexpr int OFF_B = OFF_OP + CGRP * 2 * OP_BYTES;            // [K][hi,lo]
    static constexpr int SMEM = OFF_B + ((2 * K * B_BYTES + 1023) & ~1023);
};

template <int K>
struct TcW {
    float w[K * K * K];
};

struct TcArgs {
    float* dst;
    int nx, ny, nz;
    int items_x, items_y, items_z, nitems, zchunk;   // items: x, then y, then z, then volume
    int64_t vs_dst;      // voxels from one volume's destination to the next
    int wexp;            // weights are scaled by 2^wexp before splitting
    unsigned* status;
};

// header of the shared memory map (first 1024 bytes)
struct TcHeader {
    uint64_t stage_full[STAGES];
    uint64_t stage_empty[STAGES];
    uint64_t op_full[CGRP];
    uint64_t op_empty[CGRP];
    uint64_t d_full[3];
    uint64_t d_free[3];
    uint64_t drain;
    uint32_t tmem_base;
    int abort_flag;
    int sc[SC_RING];     // per-plane scale exponents written by the converters
    float red[CGRP][2][CONV_WARPS];   // converter max reduction; negative: the warp gave up
};
static_assert(sizeof(TcHeader) <= 1024, "header");

// tcgen05 shared-memory matrix descriptor, no swizzle, K-major canonical layout of 8-row x 16-byte
// core matrices.  Low word: start address and leading (K) byte offset, >> 4; high word: stride
// (M/N) byte offset 128 >> 4 and the fixed value 0b001 in its bits 14-16, the same for every operand.
constexpr uint32_t DESC_HI = (128 >> 4) | (1u << 14);
__device__ __forceinline__ uint32_t umma_desc(uint32_t saddr, uint32_t lbo)
{
    return ((saddr >> 4) & 0x3FFF) | (((lbo >> 4) & 0x3FFF) << 16);
}

template <bool ACC>
__device__ __forceinline__ void umma_f16(uint32_t dtmem, uint32_t adesc, uint32_t bdesc, uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "mov.b64 da, {%1, %5};\n\tmov.b64 db, {%2, %5};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}" ::"r"(dtmem),
        "r"(adesc), "r"(bdesc), "r"(idesc), "n"(ACC ? 1 : 0), "n"(DESC_HI)
        : "memory");
}

__device__ __forceinline__ void umma_commit(uint64_t* bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 columns of this warp's 32 lanes into v[0..15]; complete after tmem_wait_ld()
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, float* v)
{
    uint32_t* r = reinterpret_cast<uint32_t*>(v);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void named_sync(int id, int n)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Bounded wait that also gives up when another role has aborted.  The waiting thread asks
// to be suspended (up to the hint) instead of polling, so idle roles do not take issue
// slots from the MMA-issuing warp on their sub-partition.
__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                              unsigned* status)
{
    if (mbar_try_wait_sleep(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    while (!mbar_try_wait_sleep(bar, parity)) {
        if (*abort_flag) return false;
        if (global_ns() - t0 > WAIT_LIMIT_NS) {
            *abort_flag = 1;
            atomicOr(status, STATUS_TIMEOUT);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }

template <int K>
__global__ void __launch_bounds__(NTHREADS, 1)
    k_tc(const __grid_constant__ CUtensorMap tmap, const TcArgs p, const TcW<K> W)
{
    using C = TcCfg<K>;
    constexpr int R = C::R, N = C::N;
    extern __shared__ __align__(1024) unsigned char smem[];
    TcHeader& h = *reinterpret_cast<TcHeader*>(smem);
    volatile int* abort_flag = &h.abort_flag;
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;

    // ---- set-up: barriers, TMEM, Toeplitz operands
    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&h.stage_full[s], 1);
            mbar_init(&h.stage_empty[s], 1);
        }
        for (int b = 0; b < CGRP; ++b) {
            mbar_init(&h.op_full[b], CONV_WARPS);
            mbar_init(&h.op_empty[b], 1);
        }
        for (int b = 0; b < C::DBUF; ++b) {
            mbar_init(&h.d_full[b], 2);          // MMA completion + the issuer's scale hand-off
            mbar_init(&h.d_free[b], NEPI / 32);
        }
        mbar_init(&h.drain, 1);
        h.abort_flag = 0;
        fence_mbar_init();
        prefetch_tensor_map(&tmap);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&h.tmem_base)),
                     "r"(C::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    {
        // T_b hi/lo, K-major [kc][n][8 halves] with n = (slot c, j) and entry kk = kc*8 + e.
        // STACK: 2N rows per kc chunk, the hi matrix's first; otherwise the hi matrix, then the lo matrix.
        const float sw = pow2f(p.wexp);
        __half* B = reinterpret_cast<__half*>(smem + C::OFF_B);
        const int per_b = 2 * N * 8;
        for (int i = tid; i < K * per_b; i += NTHREADS) {
            const int b = i / per_b, rem = i - b * per_b;
            const int kc = rem / (N * 8), n = (rem / 8) % N, e = rem % 8;
            const int c = n / 8, j = n % 8, kk = kc * 8 + e;
            const int a = kk - j - 4 + R;
            float v = 0.f;
            if (c < K && a >= 0 && a < K) v = W.w[(c * K + b) * K + a] * sw;
            const __half hi = __float2half_rn(v);
            const __half lo = __float2half_rn(v - __half2float(hi));
            __half* Bb = B + 2 * b * (C::B_BYTES / 2);
            if (C::STACK) {
                Bb[(kc * 2 * N + n) * 8 + e] = hi;
                Bb[(kc * 2 * N + N + n) * 8 + e] = lo;
            } else {
                Bb[rem] = hi;
                Bb[C::B_BYTES / 2 + rem] = lo;
            }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = h.tmem_base;
    const uint32_t sbase = smem_u32(smem);

    if (warp >= EPI_WARP0) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_EPI));
        // ---------------- epilogue
        const int et = tid - EPI_WARP0 * 32;            // 0..255
        const int t = et / 128;                          // x tile
        const int quad = warp & 3;                       // TMEM lane quadrant of this warp
        const int m = quad * 32 + lane;                  // output row within the tile
        const uint32_t lane_addr = static_cast<uint32_t>(quad * 32) << 16;
        uint32_t g = 0;
        float2 acc[K][4];
        bool ok = true;
        for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
            const int xi = item % p.items_x, yi = (item / p.items_x) % p.items_y;
            const int zv = item / (p.items_x * p.items_y);
            const int vol = zv / p.items_z, zi = zv - vol * p.items_z;
            float* const dst = p.dst + vol * p.vs_dst;
            const int x0 = xi * 8 * XT, y0 = yi * MROWS, zc0 = zi * p.zchunk;
            const int zc1 = min(zc0 + p.zchunk, p.nz);
            const int nplanes = zc1 - zc0 + 2 * R;
            const int oy = y0 + m, ox = x0 + 8 * t;
            const int nvalid = p.nx - ox;
#pragma unroll
            for (int c = 0; c < K; ++c)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[c][j] = make_float2(0.f, 0.f);

            auto plane = [&](const int it, const int u) {
                const int db = g % C::DBUF;
                int w = 1;
                if (lane == 0) w = wait_or_abort(&h.d_full[db], (g / C::DBUF) & 1, abort_flag, p.status) ? 1 : 0;
                w = __shfl_sync(0xffffffffu, w, 0);
                if (!w) {
                    ok = false;
                    return;
                }
                tc_fence_after();
                const float inv = pow2f(-(h.sc[g % SC_RING] + p.wexp));
                const uint32_t col = tbase + lane_addr + static_cast<uint32_t>((db * XT + t) * C::DN);
                // two 16-column loads in flight per wait: slots 4q .. 4q+3, or both parts of 2q and 2q+1
                constexpr int SPL = C::STACK ? 2 : 4;
#pragma unroll
                for (int q = 0; q < (C::SLOTS + SPL - 1) / SPL; ++q) {
                    float d[32];
                    const bool two = C::STACK || 2 * q + 1 < N / 16;
                    tmem_ld16_nowait(col + 8 * SPL * q, d);
                    if (two) tmem_ld16_nowait(col + 8 * SPL * q + (C::STACK ? N : 16), d + 16);
                    tmem_wait_ld();
#pragma unroll
                    for (int h2 = 0; h2 < SPL; ++h2) {
                        const int c = SPL * q + h2;
                        if (c < K && (h2 < 2 || two)) {
                            const int sl = ((u - c + R) % K + K) % K;
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                float2 v = make_float2(d[8 * h2 + 2 * j], d[8 * h2 + 2 * j + 1]);
                                if (C::STACK)
                                    v = __fadd2_rn(v, make_float2(d[16 + 8 * h2 + 2 * j], d[16 + 8 * h2 + 2 * j + 1]));
                                acc[sl][j] = __ffma2_rn(v, make_float2(inv, inv), acc[sl][j]);
                            }
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&h.d_free[db]);
                const int sl0 = ((u - R) % K + K) % K;
                if (it >= 2 * R && oy < p.ny && nvalid > 0) {
                    const int oz = zc0 + it - 2 * R;
                    float* d = dst + (static_cast<int64_t>(oz) * p.ny + oy) * p.nx + ox;
                    if (nvalid >= 8 && ((reinterpret_cast<uintptr_t>(d) & 15) == 0)) {
                        reinterpret_cast<float4*>(d)[0] = make_float4(acc[sl0][0].x, acc[sl0][0].y, acc[sl0][1].x, acc[sl0][1].y);
                        reinterpret_cast<float4*>(d)[1] = make_float4(acc[sl0][2].x, acc[sl0][2].y, acc[sl0][3].x, acc[sl0][3].y);
                    } else {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (j < nvalid) d[j] = j & 1 ? acc[sl0][j / 2].y : acc[sl0][j / 2].x;
                    }
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[sl0][j] = make_float2(0.f, 0.f);
                ++g;
            };

            for (int g0 = 0; g0 < nplanes && ok; g0 += K) {
#pragma unroll
                for (int u = 0; u < K; ++u) {
                    if (g0 + u >= nplanes || !ok) break;
                    plane(g0 + u, u);
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_CONV));
        if (warp == TMA_WARP) {
            // ---------------- TMA producer
            if (lane == 0) {
                uint32_t g = 0;
                bool ok = true;
                for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
                    const int xi = item % p.items_x, yi = (item / p.items_x) % p.items_y;
                    const int zv = item / (p.items_x * p.items_y);
                    const int vol = zv / p.items_z, zi = zv - vol * p.items_z;
                    const int x0 = xi * 8 * XT, y0 = yi * MROWS, zc0 = zi * p.zchunk;
                    const int zc1 = min(zc0 + p.zchunk, p.nz);
                    const int nplanes = zc1 - zc0 + 2 * R;
                    for (int it = 0; it < nplanes; ++it, ++g) {
                        const int s = g % STAGES;
                        if (g >= STAGES && !wait_or_abort(&h.stage_empty[s], ((g / STAGES) - 1) & 1,
                                                          abort_flag, p.status)) {
                            ok = false;
                            break;
                        }
                        mbar_arrive_expect_tx(&h.stage_full[s], C::STAGE_TX);
                        tma_load_4d(smem + C::OFF_STAGE + s * C::STAGE_BYTES, &tmap, &h.stage_full[s],
                                    x0 - 4, y0 - R, clampi(zc0 - R + it, 0, p.nz - 1), vol);
                    }
                }
                // drain: every issued load completes its stage (bounded, no abort check)
                for (uint32_t q = (g > STAGES ? g - STAGES : 0); q < g; ++q)
                    mbar_wait(&h.stage_full[q % STAGES], (q / STAGES) & 1);
            }
        } else if (warp == MMA_WARP) {
            // ---------------- MMA issuer: lane 0 issues, the warp walks the planes together
            {
                // idesc: D f32, A f16, B f16, both K-major, N >> 3 at bit 17, M >> 4 at bit 24
                auto idesc_of = [](int n) {
                    return (1u << 4) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(MROWS >> 4) << 24);
                };
                const uint32_t idesc = idesc_of(N), idesc2 = idesc_of(2 * N);
                // Each MMA adds a compile-time offset to the start address field of two bases (addresses
                // stay below 256 KB, so the add never carries out).
                const uint32_t a0 = umma_desc(sbase + C::OFF_OP, C::CHUNK_BYTES);
                const uint32_t b0 = umma_desc(sbase + C::OFF_B, (C::STACK ? 2 : 1) * N * 16);
                const uint32_t tb = __shfl_sync(0xffffffffu, tbase, 0);
                uint32_t g = 0;
                bool ok = true;
                for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
                    const int zi = item / (p.items_x * p.items_y) % p.items_z;
                    const int zc0 = zi * p.zchunk, zc1 = min(zc0 + p.zchunk, p.nz);
                    const int nplanes = zc1 - zc0 + 2 * R;
                    for (int it = 0; it < nplanes; ++it, ++g) {
                        const uint32_t ob = g % CGRP, db = g % C::DBUF;
                        int w = 1;
                        if (lane == 0)
                            w = wait_or_abort(&h.op_full[ob], (g / CGRP) & 1, abort_flag, p.status) &&
                                (g < C::DBUF || wait_or_abort(&h.d_free[db], ((g / C::DBUF) - 1) & 1, abort_flag, p.status));
                        if (!__shfl_sync(0xffffffffu, w, 0)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        if (lane == 0) {
                            mbar_arrive(&h.d_full[db]);   // early: hands the plane's scale on to the epilogue
                            const uint32_t ahi = a0 + ob * (2 * C::OP_BYTES >> 4), alo = ahi + (C::OP_BYTES >> 4);
                            const uint32_t d0 = tb + db * (XT * C::DN);
                            // (opaque, or the sums below are kept across planes and spilled)
                            uint32_t b1 = b0;
                            asm volatile("" : "+r"(b1));
#pragma unroll
                            for (int t = 0; t < XT; ++t) {
#pragma unroll
                                for (int b = 0; b < K; ++b) {
                                    const uint32_t ao = (t * C::CHUNK_BYTES + b * 16) >> 4;
                                    const uint32_t bh = b1 + (2 * b * C::B_BYTES >> 4), bl = bh + (C::B_BYTES >> 4);
                                    const uint32_t dt = d0 + t * C::DN;
                                    if (C::STACK) {
                                        if (b == 0)
                                            umma_f16<false>(dt, ahi + ao, bh, idesc2);
                                        else
                                            umma_f16<true>(dt, ahi + ao, bh, idesc2);
                                    } else {
                                        if (b == 0)
                                            umma_f16<false>(dt, ahi + ao, bh, idesc);
                                        else
                                            umma_f16<true>(dt, ahi + ao, bh, idesc);
                                        umma_f16<true>(dt, ahi + ao, bl, idesc);
                                    }
                                    umma_f16<true>(dt, alo + ao, bh, idesc);
                                }
                            }
                            if (C::STACK) umma_commit(&h.op_empty[ob]);
                            umma_commit(&h.d_full[db]);
                        }
                        __syncwarp();
                    }
                }
                // drain: all MMAs issued so far complete before TMEM is released
                if (lane == 0) {
                    umma_commit(&h.drain);
                    mbar_wait(&h.drain, 0);
                }
            }
        } else if (warp < EPI_WARP0 && warp % 4 != MMA_WARP) {
            // ---------------- converters: f32 tile -> fp16 hi/lo operand planes
            // Group gr converts every third plane into operand buffer gr, while the MMAs read the others:
            // the MMAs keep shared memory busy, so each step here takes a good part of a plane's time.
            // Loading, scaling and splitting wait for the stage only.
            const int gr = warp / 4;
            const int cw = max(warp % 4 - 1, 0);            // the warp's chunk
            const bool first = cw == 0 && lane == 0;        // of the group
            // items: (row, half) with the half fastest, so that a quarter warp's 16-byte reads of the
            // stage (rows 96 bytes apart) and its 8-byte writes of the operand planes touch distinct banks
            const int half = lane & 1;
            const bool extra = lane < C::EXTRA;             // one more: row 128 + lane / 2
            unsigned char* const ohi = smem + C::OFF_OP + (2 * gr + 0) * C::OP_BYTES + cw * C::CHUNK_BYTES;
            unsigned char* const olo = smem + C::OFF_OP + (2 * gr + 1) * C::OP_BYTES + cw * C::CHUNK_BYTES;
            uint32_t g = 0;
            bool ok = true, gone = false;
            for (int item = blockIdx.x; item < p.nitems && ok; item += gridDim.x) {
                const int xi = item % p.items_x, yi = (item / p.items_x) % p.items_y;
                const int zi = item / (p.items_x * p.items_y) % p.items_z;
                const int x0 = xi * 8 * XT, y0 = yi * MROWS, zc0 = zi * p.zchunk;
                const int zc1 = min(zc0 + p.zchunk, p.nz);
                const int nplanes = zc1 - zc0 + 2 * R;
                // Rows are whole 16 bytes, so the lane's 4 columns are inside the volume together or
                // outside it together; outside they repeat the first or the last column.
                const int gx0 = x0 - 4 + 8 * cw + 4 * half;
                const bool left = gx0 < 0, right = gx0 >= p.nx;
                const int col = left ? 4 : right ? p.nx - x0 : 8 * cw + 4 * half;   // in the tile
                const int ymax = p.ny - 1 - (y0 - R), ymin = R - y0;    // rows of the tile inside the volume
                for (int it = 0; it < nplanes; ++it, ++g) {
                    if (static_cast<int>(g % CGRP) != gr) continue;
                    const int s = g % STAGES;
                    int w = gone ? 0 : 1;
                    if (lane == 0 && !gone)
                        w = wait_or_abort(&h.stage_full[s], (g / STAGES) & 1, abort_flag, p.status) ? 1 : 0;
                    w = __shfl_sync(0xffffffffu, w, 0);
                    const float* st = reinterpret_cast<const float*>(smem + C::OFF_STAGE + s * C::STAGE_BYTES);
                    float v[C::MAIN + 1][4];
                    float mx = 0.f;
                    auto fetch = [&](float (&o)[4], int row) {
                        const float* sr = st + min(max(row, ymin), ymax) * (NCH * 8);
                        const float4 a = *reinterpret_cast<const float4*>(sr + col);
                        o[0] = right ? a.w : a.x;
                        o[1] = left ? a.x : right ? a.w : a.y;
                        o[2] = left ? a.x : right ? a.w : a.z;
                        o[3] = left ? a.x : a.w;
#pragma unroll
                        for (int e = 0; e < 4; ++e) mx = fmaxf(mx, fabsf(o[e]));
                    };
                    if (w) {
#pragma unroll
                        for (int q = 0; q < C::MAIN; ++q) fetch(v[q], 16 * q + lane / 2);
                        if (extra) fetch(v[C::MAIN], MROWS + lane / 2);
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                    float* red = h.red[gr][(g / CGRP) & 1];
                    if (lane == 0) red[cw] = w ? mx : -1.f;
                    named_sync(1 + gr, NCONV);
                    const float r0 = red[0], r1 = red[1], r2 = red[2];
                    if (fminf(fminf(r0, r1), r2) < 0.f) {   // the group gives up together
                        ok = false;
                        break;
                    }
                    if (first) mbar_arrive(&h.stage_empty[s]);
                    mx = fmaxf(fmaxf(r0, r1), r2);
                    // scale exponent: max|x| * 2^e in [2^13, 2^14)
                    int e = 0;
                    if (mx > 0.f && mx <= 3.0e38f) e = min(max(140 - (__float_as_int(mx) >> 23), -100), 100);
                    const float sx = pow2f(e);
                    uint2 hi[C::MAIN + 1], lo[C::MAIN + 1];
#pragma unroll
                    for (int q = 0; q <= C::MAIN; ++q) {
                        if (q == C::MAIN && !extra) continue;
                        uint32_t hw[2], lw[2];
#pragma unroll
                        for (int e2 = 0; e2 < 2; ++e2) {
                            const float2 a = __fmul2_rn(make_float2(v[q][2 * e2], v[q][2 * e2 + 1]), make_float2(sx, sx));
                            const __half2 ah = __floats2half2_rn(a.x, a.y);
                            const float2 af = __half22float2(ah);
                            const float2 al = __ffma2_rn(af, make_float2(-1.f, -1.f), a);
                            const __half2 ll = __floats2half2_rn(al.x, al.y);
                            hw[e2] = *reinterpret_cast<const uint32_t*>(&ah);
                            lw[e2] = *reinterpret_cast<const uint32_t*>(&ll);
                        }
                        hi[q] = make_uint2(hw[0], hw[1]);
                        lo[q] = make_uint2(lw[0], lw[1]);
                    }
                    // the MMAs of the buffer's last plane are done (a warp that gives up here takes the
                    // group out at its next plane)
                    w = 1;
                    if (g >= CGRP) {
                        if (lane == 0)
                            // (three D buffers: plane g's barrier is the one that plane g - 3 completes next)
                            w = wait_or_abort(C::STACK ? &h.op_empty[gr] : &h.d_full[gr], ((g / CGRP) - 1) & 1, abort_flag,
                                              p.status) ? 1 : 0;
                        w = __shfl_sync(0xffffffffu, w, 0);
                    }
                    if (!w) {
                        gone = true;
                        continue;
                    }
#pragma unroll
                    for (int q = 0; q <= C::MAIN; ++q) {
                        if (q == C::MAIN && !extra) continue;
                        *reinterpret_cast<uint2*>(ohi + q * 256 + lane * 8) = hi[q];
                        *reinterpret_cast<uint2*>(olo + q * 256 + lane * 8) = lo[q];
                    }
                    if (first) h.sc[g % SC_RING] = e;
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&h.op_full[gr]);
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase),
                     "r"(C::TMEM_COLS)
                     : "memory");
    }
}

// The kernel's warpgroups hand registers on: it must have been built with as many as they count on.
// Where it was not, tensor_available says so and a call that may choose takes the direct path.
// (Without a device there is no answer, and no launch either.)
template <int K>
bool registers_fit()
{
    static const bool fit = [] {
        cudaFuncAttributes fa{};
        if (cudaFuncGetAttributes(&fa, k_tc<K>) == cudaSuccess) return fa.numRegs >= REGS;
        cudaGetLastError();
        return true;
    }();
    return fit;
}

template <int K>
vktError launch_k(const Job& job, const float* w, const Ctx& ctx)
{
    using C = TcCfg<K>;
    TcArgs a;
    a.dst = static_cast<float*>(job.dst);
    a.nx = job.nx;
    a.ny = job.ny;
    a.nz = job.nz;
    a.status = ctx.status;
    TcW<K> W;
    float mx = 0.f;
    for (int i = 0; i < K * K * K; ++i) {
        W.w[i] = w[i];
        mx = std::max(mx, std::fabs(w[i]));
    }
    int ex = 0;
    if (mx > 0.f && std::isfinite(mx)) std::frexp(mx, &ex);
    a.wexp = (mx > 0.f && std::isfinite(mx)) ? std::min(std::max(14 - ex, -100), 100) : 0;

    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess)
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    a.items_x = (job.nx + 8 * XT - 1) / (8 * XT);
    a.items_y = (job.ny + MROWS - 1) / MROWS;
    const int nvol = std::max(job.nvol, 1);
    const long xy = static_cast<long>(a.items_x) * a.items_y;
    // whole waves of one CTA per SM over all volumes' items, counting each chunk's halo planes
    a.zchunk = zchunk_waves(xy * nvol, job.nz, sms, C::R);
    a.items_z = (job.nz + a.zchunk - 1) / a.zchunk;
    if (xy * a.items_z > 0x7fffffff / nvol) return VKT_ERROR_UNSUPPORTED;
    a.nitems = static_cast<int>(xy * a.items_z * nvol);
    a.vs_dst = job.vs_dst;

    alignas(64) CUtensorMap map;
    if (!encode_tensor_map(&map, FMT_F32, job.src, job.nx, job.ny, job.nz, nvol, job.vs_src, NCH * 8,
                           C::ROWS, 1))
        return VKT_ERROR_UNSUPPORTED;
    cudaError_t e = cudaFuncSetAttribute(k_tc<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e != cudaSuccess) return from_cuda(e);
    if (!registers_fit<K>()) return VKT_ERROR_UNSUPPORTED;
    const int grid = static_cast<int>(std::min<long>(a.nitems, sms));
    if (ctx.debug & VKT_DEBUG_LOG)
        fprintf(stderr, "[vkt] tensor k=%d items=%d (%dx%dx%d, zchunk %d) grid=%d smem=%d\n", K,
                a.nitems, a.items_x, a.items_y, a.items_z, a.zchunk, grid, C::SMEM);
    k_tc<K><<<grid, NTHREADS, C::SMEM, ctx.stream>>>(map, a, W);
    count_launches(1);
    return from_cuda(cudaGetLastError());
}

}  // namespace

vktError tensor_available(const vktStructuredVolume_impl* dst, const vktStructuredVolume_impl* src,
                          const vktFilter_impl* f)
{
    if (src->format != vktDataFormatFloat32 || dst->format != vktDataFormatFloat32)
        return VKT_ERROR_UNSUPPORTED;
    if (f->k != 5 && f->k != 7 && f->k != 9) return VKT_ERROR_UNSUPPORTED;
    if (src->dims[0] % 4 != 0 || reinterpret_cast<uintptr_t>(src->data) % 16 != 0)
        return VKT_ERROR_UNSUPPORTED;   // rows must be describable by a TMA tensor map
    if (!(f->k == 5 ? registers_fit<5>() : f->k == 7 ? registers_fit<7>() : registers_fit<9>()))
        return VKT_ERROR_UNSUPPORTED;
    return VKT_NO_ERROR;
}

bool tensor_batchable(const Job& job, int32_t n, int64_t vs)
{
    // the tensor map's volume stride is a multiple of 16 bytes, and the items are counted in 31 bits
    const int64_t items = static_cast<int64_t>((job.nx + 15) / 16) * ((job.ny + MROWS - 1) / MROWS) * job.nz;
    return (vs * 4) % 16 == 0 && items <= 0x7fffffff / n;
}

vktError launch_tensor(const Job& job, const float* w, int k, const Ctx& ctx)
{
    switch (k) {
    case 5: return launch_k<5>(job, w, ctx);
    case 7: return launch_k<7>(job, w, ctx);
    case 9: return launch_k<9>(job, w, ctx);
    default: return VKT_ERROR_UNSUPPORTED;
    }
}

}  // namespace vkt
