// vkt_render.cu -- headless Render: volume ray marching with absorption and emission (Sec.
// 3.2 "Rendering", classified by an RGBA lookup table), one thread per pixel, into a device
// RGBA float image (no window, no graphics API).
//
// World coordinates are voxel units: the volume is the box [0,nx] x [0,ny] x [0,nz] with
// voxel (i,j,k) centred at (i+0.5, j+0.5, k+0.5).  A pinhole camera casts one ray per pixel
// centre; the ray enters the box at t0 (slab test, clamped to t >= 0) and is sampled at
// t0 + (k + 0.5) * step while inside.  A sample is the trilinear blend of the stored voxels
// (clamped at the faces), normalised by the volume's value range to u in [0,1], classified
// by the linearly blended table entry at u (n entries at i/(n-1), straight colours), its
// opacity corrected to the step (1 - (1 - a)^step), and composited front to back; a ray
// stops once its opacity reaches the termination value.  The table lives in shared memory.
//
// Bound by issue (about 108 instructions per sample, 89 % of the slots) and, where a warp's rays lie
// on many voxel rows, by the gathers' cache accesses.  Against the first: 32-bit offsets, an inside
// path without clamps, conversions by bit pattern (eight conversions per sample would keep the
// conversion unit as busy as the issue slots), table entries with their differences; against the
// second: the shape of a warp's pixel tile (tile_of) and a cell's voxels kept from sample to sample
// (REUSE_ROWS).  1024 x 768 of a 512^3 uint8 volume, step 0.5: 1572 -> 1223 us a frame.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <type_traits>

#include "vkt_internal.h"

namespace vkt {
namespace {

constexpr int BX = 16, BY = 16;

struct RenderArgs {
    const void* src;
    int fmt;
    int nx, ny, nz;
    int64_t row_bytes, plane_bytes;
    float lo, hi, qinv;          // qinv = 1 / (2^N - 1) for integer formats
    int width, height;
    float eye[3], f[3], r[3], u[3];
    float th, aspect;            // tan(fovy / 2), width / height
    float step, termination;
    float bg[4];
    int tile;                    // a warp's tile is 2^tile pixels wide
    int lut_n;
    float lut[VKT_RENDER_MAX_LUT * 4];
};

template <int FMT, typename Off>
__device__ __forceinline__ float voxel(const void* src, Off i)
{
    if constexpr (FMT == vktDataFormatUint8) return static_cast<float>(__ldg(static_cast<const uint8_t*>(src) + i));
    else if constexpr (FMT == vktDataFormatUint16) return static_cast<float>(__ldg(static_cast<const uint16_t*>(src) + i));
    else return __ldg(static_cast<const float*>(src) + i);
}

// The voxel at `at` and its neighbour along x, as their blend needs them: (v0, v1) of a float
// volume, whose voxels may be infinite, else (v0, v1 - v0).  A code q is read as the float 2^23 + q,
// whose bits are q's in the mantissa: the difference of two is exact, and one more subtraction
// gives v0 (the conversion unit runs at an eighth of the rate of these).
template <int FMT>
__device__ __forceinline__ float2 pair_x(const void* at)
{
    if constexpr (FMT == vktDataFormatFloat32) {
        const float* v = static_cast<const float*>(at);
        return make_float2(__ldg(v), __ldg(v + 1));
    } else {
        uint32_t q0, q1;
        if constexpr (FMT == vktDataFormatUint8) {
            q0 = __ldg(static_cast<const uint8_t*>(at));
            q1 = __ldg(static_cast<const uint8_t*>(at) + 1);
        } else {
            q0 = __ldg(static_cast<const uint16_t*>(at));
            q1 = __ldg(static_cast<const uint16_t*>(at) + 1);
        }
        const float b0 = __uint_as_float(q0 | 0x4B000000u), b1 = __uint_as_float(q1 | 0x4B000000u);
        return make_float2(b0 - 8388608.f, b1 - b0);
    }
}

template <int FMT>
__device__ __forceinline__ float blend_x(float2 v, float w)
{
    return FMT == vktDataFormatFloat32 ? v.x * (1.f - w) + v.y * w : fmaf(w, v.y, v.x);
}

// The eight voxels around a sample, kept from one sample of a ray to the next (REUSE): where a
// warp's rays lie on many voxel rows, the gathers are what a sample costs most, and rays that
// stay in their cell need none (REUSE_ROWS).
template <typename Off>
struct Cell {
    Off at = static_cast<Off>(-1);   // offset of the lowest voxel; -1: none
    float2 v[4];                     // rows (y, z) (y + 1, z) (y, z + 1) (y + 1, z + 1)
};

// x's cell along one axis, the integer i at or below x, and w = x - i: x is rounded down to an integer
// in the low bits of 1.5 * 2^23 + x.  (At a whole x the blend has to take that voxel with weight 1 and
// the one above it with 0: 0 times an infinite voxel is NaN, so the cell below would not do.)
// BIG: axes of more than 2^21 voxels, where that has too few bits.
template <bool BIG>
__device__ __forceinline__ int cell(float x, float& w)
{
    if constexpr (BIG) {
        const float f = floorf(x);
        w = x - f;
        return static_cast<int>(f);
    }
    const float s = __fadd_rd(x, 12582912.f);
    w = x - (s - 12582912.f);
    return static_cast<int>(__float_as_uint(s)) - 0x4B400000;
}

// u in [0,1] of the sample at x, y, z (in voxels from the centre of voxel 0): trilinear blend of
// the stored voxels, clamped at the faces, then the range map.
// Off: the type of voxel offsets (32 bits for volumes under 2^32 voxels: fewer address
// instructions per gather, 14 % faster per frame)
template <int FMT, typename Off, bool REUSE>
__device__ __forceinline__ float sample_u(const RenderArgs& a, float x, float y, float z, Cell<Off>& c)
{
    float wx, wy, wz;
    constexpr bool BIG = sizeof(Off) == 8;
    const int ix = cell<BIG>(x, wx), iy = cell<BIG>(y, wy), iz = cell<BIG>(z, wz);
    float s;
    if (static_cast<unsigned>(ix) < static_cast<unsigned>(a.nx - 1) &&
        static_cast<unsigned>(iy) < static_cast<unsigned>(a.ny - 1) &&
        static_cast<unsigned>(iz) < static_cast<unsigned>(a.nz - 1)) {
        // all eight voxels inside: one offset, the other rows at fixed distances
        const Off i = (static_cast<Off>(iz) * a.ny + iy) * a.nx + ix;
        if (!REUSE || i != c.at) {
            c.at = i;
            constexpr int ES = FMT == vktDataFormatUint8 ? 1 : FMT == vktDataFormatUint16 ? 2 : 4;
            const unsigned char* q = static_cast<const unsigned char*>(a.src) + static_cast<uint64_t>(i) * ES;
            c.v[0] = pair_x<FMT>(q);
            c.v[1] = pair_x<FMT>(q + a.row_bytes);
            q += a.plane_bytes;
            c.v[2] = pair_x<FMT>(q);
            c.v[3] = pair_x<FMT>(q + a.row_bytes);
        }
        const float c00 = blend_x<FMT>(c.v[0], wx), c01 = blend_x<FMT>(c.v[1], wx);
        const float c10 = blend_x<FMT>(c.v[2], wx), c11 = blend_x<FMT>(c.v[3], wx);
        if constexpr (FMT == vktDataFormatFloat32) {
            const float c0 = c00 * (1.f - wy) + c01 * wy, c1 = c10 * (1.f - wy) + c11 * wy;
            s = c0 * (1.f - wz) + c1 * wz;
        } else {
            const float c0 = fmaf(wy, c01 - c00, c00), c1 = fmaf(wy, c11 - c10, c10);
            s = fmaf(wz, c1 - c0, c0);
        }
    } else {
        const int x0 = min(max(ix, 0), a.nx - 1), x1 = min(max(ix + 1, 0), a.nx - 1);
        const int y0 = min(max(iy, 0), a.ny - 1), y1 = min(max(iy + 1, 0), a.ny - 1);
        const int z0 = min(max(iz, 0), a.nz - 1), z1 = min(max(iz + 1, 0), a.nz - 1);
        const Off pz0 = static_cast<Off>(z0) * a.ny, pz1 = static_cast<Off>(z1) * a.ny;
        const Off r00 = (pz0 + y0) * a.nx, r01 = (pz0 + y1) * a.nx;
        const Off r10 = (pz1 + y0) * a.nx, r11 = (pz1 + y1) * a.nx;
        const float c00 = voxel<FMT>(a.src, r00 + x0) * (1.f - wx) + voxel<FMT>(a.src, r00 + x1) * wx;
        const float c01 = voxel<FMT>(a.src, r01 + x0) * (1.f - wx) + voxel<FMT>(a.src, r01 + x1) * wx;
        const float c10 = voxel<FMT>(a.src, r10 + x0) * (1.f - wx) + voxel<FMT>(a.src, r10 + x1) * wx;
        const float c11 = voxel<FMT>(a.src, r11 + x0) * (1.f - wx) + voxel<FMT>(a.src, r11 + x1) * wx;
        const float c0 = c00 * (1.f - wy) + c01 * wy, c1 = c10 * (1.f - wy) + c11 * wy;
        s = c0 * (1.f - wz) + c1 * wz;
    }
    // integer codes: v = lo + (hi - lo) s / qmax, so u = s / qmax; float voxels: u = (s - lo)/(hi - lo)
    if constexpr (FMT == vktDataFormatFloat32) return __saturatef((s - a.lo) / (a.hi - a.lo));
    return __saturatef(s * a.qinv);
}

// 2^x and log2(x) by the hardware's approximations with denormal results as 0, which 1 - 2^x and
// log2(1 - a) (a multiple of 2^-24) cannot tell
__device__ __forceinline__ float exp2_ftz(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float log2_ftz(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int FMT, typename Off, bool REUSE>
__global__ void __launch_bounds__(BX* BY) k_render(const __grid_constant__ RenderArgs a, float* __restrict__ rgba)
{
    // entry i and its difference to the next (GENERAL: the next itself, which may be infinite); the
    // last entry's next is itself, since fi = n - 1 lies in cell n - 1 with w = 0
    constexpr bool GENERAL = sizeof(Off) == 8;
    __shared__ float4 lut[VKT_RENDER_MAX_LUT][2];
    const int tid = threadIdx.y * BX + threadIdx.x;
    for (int i = tid; i < a.lut_n; i += BX * BY) {
        const float* e = a.lut + 4 * i;
        const float* n = a.lut + 4 * min(i + 1, a.lut_n - 1);
        lut[i][0] = make_float4(e[0], e[1], e[2], e[3]);
        lut[i][1] = GENERAL ? make_float4(n[0], n[1], n[2], n[3])
                            : make_float4(n[0] - e[0], n[1] - e[1], n[2] - e[2], n[3] - e[3]);
    }
    __syncthreads();
    // a warp takes a tile of 2^tile x 2^(5 - tile) pixels of the block (tile_of)
    const int warp = tid >> 5, lane = tid & 31;
    const int across = 4 - a.tile;   // log2 of the warps side by side in a block
    const int px = blockIdx.x * BX + ((warp & ((1 << across) - 1)) << a.tile) + (lane & ((1 << a.tile) - 1));
    const int py = blockIdx.y * BY + ((warp >> across) << (5 - a.tile)) + (lane >> a.tile);
    if (px >= a.width || py >= a.height) return;

    const float sx = (2.f * (px + 0.5f) / a.width - 1.f) * a.th * a.aspect;
    const float sy = (1.f - 2.f * (py + 0.5f) / a.height) * a.th;
    float d[3];
    for (int c = 0; c < 3; ++c) d[c] = a.f[c] + sx * a.r[c] + sy * a.u[c];
    const float dn = rsqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
    for (int c = 0; c < 3; ++c) d[c] *= dn;

    const float box[3] = {static_cast<float>(a.nx), static_cast<float>(a.ny), static_cast<float>(a.nz)};
    float tn = -INFINITY, tf = INFINITY;
    bool hit = true;
    for (int c = 0; c < 3; ++c) {
        if (fabsf(d[c]) < 1e-12f) {
            if (a.eye[c] < 0.f || a.eye[c] > box[c]) hit = false;
            continue;
        }
        float ta = (0.f - a.eye[c]) / d[c], tb = (box[c] - a.eye[c]) / d[c];
        if (ta > tb) {
            const float t = ta;
            ta = tb;
            tb = t;
        }
        tn = fmaxf(tn, ta);
        tf = fminf(tf, tb);
    }
    const float t0 = fmaxf(tn, 0.f), t1 = tf;
    float C0 = 0.f, C1 = 0.f, C2 = 0.f, A = 0.f;
    if (hit && t0 < t1) {
        const float m = static_cast<float>(a.lut_n - 1);
        // positions in voxels from the centre of voxel 0
        const float ex = a.eye[0] - 0.5f, ey = a.eye[1] - 0.5f, ez = a.eye[2] - 0.5f;
        Cell<Off> near;
        for (int k = 0;; ++k) {
            const float t = t0 + (static_cast<float>(k) + 0.5f) * a.step;
            if (!(t < t1)) break;
            const float un = sample_u<FMT, Off, REUSE>(a, ex + t * d[0], ey + t * d[1], ez + t * d[2], near);
            float w;
            const float fi = un * m;       // in [0, m], so its cell is in [0, m]
            int i0 = cell<false>(fi, w);
            if constexpr (GENERAL) {       // the last entry is the upper end of the cell before it
                i0 = min(i0, a.lut_n - 2);
                w = fi - static_cast<float>(i0);
            }
            const float4 e = lut[i0][0], n = lut[i0][1];
            float cr, cg, cb, ca;
            if constexpr (GENERAL) {
                cr = e.x * (1.f - w) + n.x * w;
                cg = e.y * (1.f - w) + n.y * w;
                cb = e.z * (1.f - w) + n.z * w;
                ca = e.w * (1.f - w) + n.w * w;
            } else {
                cr = fmaf(w, n.x, e.x);
                cg = fmaf(w, n.y, e.y);
                cb = fmaf(w, n.z, e.z);
                ca = fmaf(w, n.w, e.w);
            }
            // opacity corrected to the step: 1 - (1 - a)^step = 1 - 2^(step log2(1 - a))
            const float ac = 1.f - exp2_ftz(a.step * log2_ftz(1.f - ca));
            const float tw = (1.f - A) * ac;
            C0 += tw * cr;
            C1 += tw * cg;
            C2 += tw * cb;
            A += tw;
            if (A >= a.termination) break;
        }
    }
    float* o = rgba + 4 * (static_cast<int64_t>(py) * a.width + px);
    *reinterpret_cast<float4*>(o) = make_float4(C0 + (1.f - A) * a.bg[0], C1 + (1.f - A) * a.bg[1],
                                                C2 + (1.f - A) * a.bg[2], A + (1.f - A) * a.bg[3]);
}

bool valid_volume(const vktStructuredVolume_impl* v) { return v && v->magic == VKT_VOLUME_MAGIC; }

void normalize3(double* v)
{
    const double n = std::sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    for (int c = 0; c < 3; ++c) v[c] /= n;
}

// The pixel tile of a warp: 2 x 16, 4 x 8, 8 x 4 or 16 x 2.  A gather is answered one voxel row (128
// bytes of it) at a time, so the tile to take is the one whose rays lie on the fewest rows: a pixel
// to the right moves the sample `spacing` voxels along r, of which the y and z parts change the row,
// a pixel down likewise along u.  1024 x 768, 512^3 uint8, step 0.5, us a frame at 2 / 4 / 8 / 16
// pixels wide: image x along volume x 4711 / 2598 / 1602 / 1433, image y along volume x
// 1420 / 1657 / 2646 / 4715 (8 wide, for every view: 1600 and 2640); along x 8067 to 8188.
// Returns the rows of the chosen tile.
double tile_of(const double* r, const double* u, double spacing, int* tile)
{
    const double ry = spacing * std::sqrt(r[1] * r[1] + r[2] * r[2]);
    const double uy = spacing * std::sqrt(u[1] * u[1] + u[2] * u[2]);
    double best = 0.0;
    *tile = 0;
    for (int t : {4, 3, 2, 1}) {
        const double w = 1 << t, h = 32 >> t;
        const double rows = std::fmin(1.0 + (w - 1.0) * ry, w) * std::fmin(1.0 + (h - 1.0) * uy, h);
        if (*tile == 0 || rows < 0.99 * best) {
            best = rows;
            *tile = t;
        }
    }
    return best;
}

// Above how many rows per gather the kept cell (REUSE) pays for its comparison.  Step 0.5 / 1.0,
// without and with it: 2 rows 1433 -> 1442 / 757 -> 760 us (float32 1516 -> 1597), along x (27 rows)
// 8100 -> 4670 / 4040 -> 3870, oblique (20 rows) 5193 -> 3367 / 2666 -> 2270.
constexpr double REUSE_ROWS = 4.0;

}  // namespace
}  // namespace vkt

using namespace vkt;

extern "C" vktError vktRenderSV(float* rgba, int32_t width, int32_t height, vktStructuredVolume volume,
                                const vktRenderParams* params)
{
    vkt::CallRange nvtx_range("vktRenderSV");
    if (!valid_volume(volume)) return VKT_ERROR_INVALID_HANDLE;
    if (!rgba || !params || width < 1 || height < 1 || height > 65535 * BY) return VKT_ERROR_INVALID_VALUE;
    const vktRenderParams& p = *params;
    if (p.lutSize < 2 || p.lutSize > VKT_RENDER_MAX_LUT || !p.lut) return VKT_ERROR_INVALID_VALUE;
    if (!(p.step > 0.f) || !(p.fovy > 0.f && p.fovy < 3.14159f)) return VKT_ERROR_INVALID_VALUE;
    if (reinterpret_cast<uintptr_t>(rgba) % 16 != 0) return VKT_ERROR_INVALID_VALUE;
    double f[3], up[3];
    for (int c = 0; c < 3; ++c) {
        f[c] = static_cast<double>(p.center[c]) - p.eye[c];
        up[c] = p.up[c];
    }
    const double fl = std::sqrt(f[0] * f[0] + f[1] * f[1] + f[2] * f[2]);
    double r[3] = {f[1] * up[2] - f[2] * up[1], f[2] * up[0] - f[0] * up[2], f[0] * up[1] - f[1] * up[0]};
    const double rl = std::sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]);
    if (!(fl > 0.0) || !(rl > 1e-12 * fl)) return VKT_ERROR_INVALID_VALUE;   // no view direction, or up parallel to it
    if (volume->format != vktDataFormatFloat32 && volume->lo == volume->hi) return VKT_ERROR_INVALID_VALUE;
    if (volume->format == vktDataFormatFloat32 && !(volume->hi != volume->lo)) return VKT_ERROR_INVALID_VALUE;
    Ctx ctx;
    vktError err = get_context(&ctx);
    if (err != VKT_NO_ERROR) return err;

    normalize3(f);
    normalize3(r);
    const double u[3] = {r[1] * f[2] - r[2] * f[1], r[2] * f[0] - r[0] * f[2], r[0] * f[1] - r[1] * f[0]};
    RenderArgs a;
    a.src = volume->data;
    a.fmt = volume->format;
    a.nx = volume->dims[0];
    a.ny = volume->dims[1];
    a.nz = volume->dims[2];
    const int es = volume->format == vktDataFormatUint8 ? 1 : volume->format == vktDataFormatUint16 ? 2 : 4;
    a.row_bytes = static_cast<int64_t>(a.nx) * es;
    a.plane_bytes = a.row_bytes * a.ny;
    a.lo = volume->lo;
    a.hi = volume->hi;
    a.qinv = volume->format == vktDataFormatUint8 ? 1.f / 255.f : 1.f / 65535.f;
    a.width = width;
    a.height = height;
    for (int c = 0; c < 3; ++c) {
        a.eye[c] = p.eye[c];
        a.f[c] = static_cast<float>(f[c]);
        a.r[c] = static_cast<float>(r[c]);
        a.u[c] = static_cast<float>(u[c]);
    }
    a.th = static_cast<float>(std::tan(0.5 * p.fovy));
    a.aspect = static_cast<float>(static_cast<double>(width) / height);
    a.step = p.step;
    a.termination = p.termination;
    for (int c = 0; c < 4; ++c) a.bg[c] = p.background[c];
    a.lut_n = p.lutSize;
    for (int i = 0; i < p.lutSize * 4; ++i) a.lut[i] = p.lut[i];
    const dim3 block(BX, BY), grid((width + BX - 1) / BX, (height + BY - 1) / BY);
    // voxel offsets in 32 bits while every offset of the volume fits, no axis is so long that cell()
    // wants its other form, and the table is finite
    bool finite = true;
    for (int i = 0; i < p.lutSize * 4; ++i) finite = finite && std::isfinite(p.lut[i]);
    const bool off32 = finite && static_cast<uint64_t>(a.nx) * a.ny * a.nz <= 0xffffffffull &&
                       std::max(a.nx, std::max(a.ny, a.nz)) <= (1 << 21);
    // the pixel spacing in voxels at the volume's centre
    double dist = 0.0;
    for (int c = 0; c < 3; ++c) {
        const double to = 0.5 * volume->dims[c] - p.eye[c];
        dist += to * to;
    }
    const double rows = tile_of(r, u, 2.0 * a.th * std::sqrt(dist) / height, &a.tile);
    const bool reuse = rows > REUSE_ROWS;
    auto launch = [&](auto fmt) {
        constexpr int F = decltype(fmt)::value;
        if (off32 && reuse) k_render<F, uint32_t, true><<<grid, block, 0, ctx.stream>>>(a, rgba);
        else if (off32) k_render<F, uint32_t, false><<<grid, block, 0, ctx.stream>>>(a, rgba);
        else k_render<F, int64_t, false><<<grid, block, 0, ctx.stream>>>(a, rgba);
    };
    if (volume->format == vktDataFormatUint8) launch(std::integral_constant<int, vktDataFormatUint8>{});
    else if (volume->format == vktDataFormatUint16) launch(std::integral_constant<int, vktDataFormatUint16>{});
    else launch(std::integral_constant<int, vktDataFormatFloat32>{});
    count_launches(1);
    if (ctx.debug & VKT_DEBUG_LOG)
        fprintf(stderr, "[vkt] render %dx%d of %dx%dx%d step=%g grid=(%u,%u)\n", width, height, a.nx, a.ny,
                a.nz, p.step, grid.x, grid.y);
    return from_cuda(cudaGetLastError());
}
