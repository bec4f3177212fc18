// Bit transpose of a block in place by a CTA (Sec. 4.2): a thread holds 32
// words of the block in registers, so one CTA of S / 128 threads transposes
// a block of S bytes with two barriers, for every element size and every
// block size up to 64 KiB.  The one-warp transposes of shuffle.cuh need up to
// 64 words a lane for 8 KiB blocks and cannot take larger ones in place.
//
// A block of Bb elements (any multiple of 8: the shortened last block of a
// stream is transposed the same way, its bit-rows then being whole bytes but
// not whole words) becomes 8 * ES bit-rows of Bb / 8 bytes.  Thread u:
//   ES 4: elements 32 u .. 32 u + 31, word u of the 32 bit-rows;
//   ES 8: the low (u < NG) or high words of elements 32 g .. 32 g + 31, word
//         g of bit-rows 0 .. 31 or 32 .. 63 (NG groups, g = u mod NG);
//   ES 2: elements 64 u .. 64 u + 63, words 2 u and 2 u + 1 of 16 bit-rows;
//   ES 1: elements 128 u .. 128 u + 127, words 4 u .. 4 u + 3 of 8 bit-rows.
#pragma once

#include "shuffle.cuh"

namespace bsg {

#if defined(__CUDACC__) || defined(BSG_WARP_EMU)

// Whether a block size has this transpose for its full blocks (the words of
// a bit-row belong to one thread each).
__host__ __device__ constexpr bool cta_shape_ok(uint32_t es, uint32_t B)
{
    return B != 0 && B <= 65536u / es &&
           (es == 1 ? B % 128u == 0 : es == 2 ? B % 64u == 0 : B % 32u == 0);
}

// Whether the n samples of a block of a time-slowest cube are gathered one by
// one: its time axis is longer than half the block (any length up to 2^32 - 1).
__host__ __device__ constexpr bool cta_gather_single(uint32_t T, uint32_t n) { return T > n / 2u; }

// Threads that hold a part of a block of Bb elements (whole groups, the last
// one perhaps partial).
template <int ES>
BSG_HD uint32_t cta_units(uint32_t Bb)
{
    return ES == 1   ? (Bb + 127u) / 128u
           : ES == 2 ? (Bb + 63u) / 64u
           : ES == 4 ? (Bb + 31u) / 32u
                     : 2u * ((Bb + 31u) / 32u);
}

// A thread's 32 words of the block in registers, transposed: v[r] is what
// cta_put_rows writes.  fix(g, v) sees the words of group g before the
// transpose, v[m] being component (m + 4 (g & 7)) mod 32 (ES 4 only).
template <int ES, class Fix>
BSG_D void cta_get_rows(const uint8_t *buf, uint32_t Bb, uint32_t u, uint32_t (&v)[32], Fix fix)
{
    if (ES == 4) {
        const uint8_t *grp = buf + 128u * u;
        const uint32_t rot = u & 7u;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const uint4 q = *reinterpret_cast<const uint4 *>(grp + 16u * ((k + rot) & 7u));
            v[4 * k] = q.x;
            v[4 * k + 1] = q.y;
            v[4 * k + 2] = q.z;
            v[4 * k + 3] = q.w;
        }
        fix(u, v);
        transpose32(v);
#pragma unroll
        for (int r = 0; r < 32; r++) v[r] = rotl(v[r], 4u * rot);
    } else if (ES == 8) {
        const uint32_t NG = (Bb + 31u) / 32u, h = u >= NG ? 1u : 0u, g = u - h * NG;
        const uint8_t *grp = buf + 256u * g;
        const uint32_t rot = g & 15u;
#pragma unroll
        for (int k = 0; k < 16; k++) {
            const uint4 q = *reinterpret_cast<const uint4 *>(grp + 16u * ((k + rot) & 15u));
            v[2 * k] = h ? q.y : q.x;
            v[2 * k + 1] = h ? q.w : q.z;
        }
        // v[m] holds element (m + 2 rot) mod 32
        transpose32(v);
#pragma unroll
        for (int r = 0; r < 32; r++) v[r] = rotl(v[r], 2u * rot);
    } else if (ES == 2) {
        shuf2_read_group(buf + 128u * u, u & 7u, v);
    } else {
        shuf1_read_group(buf + 128u * u, u, v);
    }
}

// The thread's words to the bit-rows at buf, a bit-row taking the whole words
// of its groups (after a barrier that ends the reads of the elements).
template <int ES>
BSG_D void cta_put_rows(uint8_t *buf, uint32_t Bb, uint32_t u, const uint32_t (&v)[32])
{
    uint32_t *d32 = reinterpret_cast<uint32_t *>(buf);
    if (ES == 4 || ES == 8) {
        const uint32_t NG = (Bb + 31u) / 32u, h = ES == 8 && u >= NG ? 1u : 0u;
        uint32_t *p = d32 + 32u * h * NG + (u - h * NG);
#pragma unroll
        for (int r = 0; r < 32; r++, p += NG) *p = v[r];
    } else if (ES == 2) {
        shuf2_put_rows(buf, (Bb + 63u) / 64u, u, v, 0, 16);
    } else {
        shuf1_put_rows(buf, 4u * ((Bb + 127u) / 128u), u, v);
    }
}

// Whether the bit-rows of Bb elements are whole groups of words; those of a
// shortened last block need not be and are moved together (cta_pack_rows).
template <int ES>
BSG_HD bool cta_rows_whole(uint32_t Bb)
{
    return Bb % (ES == 1 ? 128u : ES == 2 ? 64u : 32u) == 0;
}

// Bit-rows of Bb / 8 bytes from the whole-word rows that cta_put_rows wrote
// (after a barrier; ends with one): byte o moves down to its place, a stretch
// of bytes at a time, loaded by every thread before any stores it.
template <int ES>
BSG_D void cta_pack_rows(uint8_t *buf, uint32_t Bb)
{
    const uint32_t G = ES == 1 ? 128u : ES == 2 ? 64u : 32u;
    const uint32_t rowb = Bb / 8u, wide = (Bb + G - 1u) / G * G / 8u;
#pragma unroll 1
    for (uint32_t b = 0; b < Bb * ES; b += blockDim.x) {
        const uint32_t o = b + threadIdx.x, r = o / rowb;
        const bool in = o < Bb * ES;
        const uint8_t x = in ? buf[r * wide + (o - r * rowb)] : 0;
        __syncthreads();
        if (in) buf[o] = x;
        __syncthreads();
    }
}

#endif  // __CUDACC__ || BSG_WARP_EMU

}  // namespace bsg
