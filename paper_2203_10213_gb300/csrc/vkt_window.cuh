// vkt_window.cuh -- the x pass's window of an integer source, read from a raw stage as aligned
// 32-bit words, for every way a stage is filled (one TMA box, row copies at any misalignment,
// plain loads).
//
// A window of K + 3 codes (four outputs) is 8 to 24 bytes: two to seven word loads and at most
// one funnel shift per word, instead of K + 3 one-element loads.  The clamp at the volume's x
// faces is a select chain on the window (clamp_window), taken only by tiles that touch a face.
#pragma once

#include "vkt_tile.cuh"

namespace vkt {

// 2^23 + code i of the packed words w, as a float's bits (exact), by a byte permute
template <int SF>
__device__ __forceinline__ uint32_t code_bits(const uint32_t* w, int i)
{
    static_assert(SF == FMT_U8 || SF == FMT_U16, "integer sources");
    if constexpr (SF == FMT_U8)
        return __byte_perm(w[i >> 2], 0x4B000000u, 0x7440u + (i & 3));
    else
        return __byte_perm(w[i >> 1], 0x4B000000u, (i & 1) ? 0x7432u : 0x7410u);
}

// codes i and i + 1 as floats, minus 2^(bits-1) if CENTRE (exact): the offset of both is taken off by
// one packed addition
template <int SF, bool CENTRE>
__device__ __forceinline__ float2 code_pair(const uint32_t* w, int i)
{
    constexpr float off = CENTRE ? 8388608.f + (SF == FMT_U8 ? 128.f : 32768.f) : 8388608.f;
    return __fadd2_rn(make_float2(__uint_as_float(code_bits<SF>(w, i)), __uint_as_float(code_bits<SF>(w, i + 1))),
                      make_float2(-off, -off));
}

// win[e] = code at raw column col + shift + e of the stage row at `row`, e < K + 3.  FIXED:
// col = 4 g + (a constant) of a TMA stage (shift 0), so the words' alignment is known at
// compile time; otherwise they are aligned with a funnel shift.
// The words read lie inside the stage row: col + K + 2 is at most TX + xa + R - 1 and a row
// has TX + 2 xa columns (xa >= 16 bytes - R codes past the window), 16 bytes more where shift
// can be nonzero.
template <int K, int SF, bool FIXED, bool CENTRE>
__device__ __forceinline__ void window(const unsigned char* row, int col, uint32_t shift,
                                       float (&win)[K + 3])
{
    constexpr int ES = fmt_bytes(SF), R = (K - 1) / 2;
    if constexpr (FIXED) {
        constexpr int O = ((fmt_xalign(SF) - R) * ES) & 3;     // byte of a word the window starts at
        constexpr int NW = (O + (K + 3) * ES + 3) / 4;
        const uint32_t* p = reinterpret_cast<const uint32_t*>(row + col * ES - O);
        uint32_t w[NW];
#pragma unroll
        for (int i = 0; i < NW; ++i) w[i] = p[i];
#pragma unroll
        for (int e = 0; e < K + 3; e += 2) {
            const float2 v = code_pair<SF, CENTRE>(w, O / ES + e);
            win[e] = v.x;
            win[e + 1] = v.y;
        }
    } else {
        constexpr int NW = ((K + 3) * ES + 3) / 4;
        const uint32_t at = (static_cast<uint32_t>(col) + shift) * ES;
        const uint32_t* p = reinterpret_cast<const uint32_t*>(row + (at & ~3u));
        const uint32_t bits = (at & 3u) * 8;
        uint32_t w[NW + 1];
#pragma unroll
        for (int i = 0; i < NW + 1; ++i) w[i] = p[i];
#pragma unroll
        for (int i = 0; i < NW; ++i) w[i] = __funnelshift_r(w[i], w[i + 1], bits);
#pragma unroll
        for (int e = 0; e < K + 3; e += 2) {
            const float2 v = code_pair<SF, CENTRE>(w, e);
            win[e] = v.x;
            win[e + 1] = v.y;
        }
    }
}

// Window of the outputs gx .. gx + 3 (gx a multiple of 4) clamped at the volume's x faces:
// positions below 0 exist only for gx == 0 (R <= 4) and repeat win[R]; positions past nx - 1
// repeat their left neighbour in the window.
template <int K>
__device__ __forceinline__ void clamp_window(float (&win)[K + 3], int gx, int nx)
{
    constexpr int R = (K - 1) / 2;
#pragma unroll
    for (int e = 0; e < R; ++e) win[e] = gx == 0 ? win[R] : win[e];
    const int last = nx - 1 - gx + R;      // the window index of voxel nx - 1
#pragma unroll
    for (int e = 1; e < K + 3; ++e) win[e] = e > last ? win[e - 1] : win[e];
}

}  // namespace vkt
