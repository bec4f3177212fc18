// LZ4 block decoder for a CTA of two warps (Sec. 4.1; the format is in
// lz4_warp.cuh), in place if the caller wants: the first warp parses the
// tokens and copies the literal runs, the second copies the matches one
// batch of sequences behind.
//
// A block's sequences are a serial chain (each token's place depends on the
// lengths before it), so one warp per block spends most of its time in the
// latency of that chain.  Literals only need the input and matches only what
// lies before them in the output, so the two kinds of copies overlap with no
// more than a barrier per batch, and an SM holds twice the warps for the same
// shared memory.  In place: a batch's output ends before the input that
// follows it (the margin that decompress_inplace_kernel's comment derives
// holds after every sequence of a valid block, and the parser ends at the first
// sequence for which it does not), so the matches of one batch never touch
// what the next one reads.
#pragma once

#include "lz4_warp.cuh"

namespace bsg {

#if defined(__CUDACC__) || defined(BSG_WARP_EMU)

constexpr uint32_t DEC_BATCH = 16;                  // sequences between two barriers
constexpr uint32_t DEC_RING_WORDS = 2u * 2u * DEC_BATCH + 2u;

// Copy of len literal bytes src[s..] -> dst[d..] by one warp, where dst may
// run over src from behind (every load of a step before its stores, as
// warp_copy_ordered): long runs in steps of 512 bytes, 16 to a lane.
BSG_D void dec_literals(uint8_t *dst, uint32_t d, const uint8_t *src, uint32_t s, uint32_t len,
                        uint32_t lane)
{
    if (len < 256) {
        warp_copy_ordered(dst, d, src, s, len, lane);
        return;
    }
    const uint32_t head = (16u - (d & 15u)) & 15u;
    warp_copy_ordered(dst, d, src, s, head, lane);
    d += head;
    s += head;
    len -= head;
    const uint32_t units = len >> 4, sh = (s & 3u) * 8u;
    const uint32_t *w = reinterpret_cast<const uint32_t *>(src) + (s >> 2);
    uint4 *o = reinterpret_cast<uint4 *>(dst + d);
#pragma unroll 1
    for (uint32_t b = 0; b < units; b += 32) {
        const uint32_t u = b + lane;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (u < units) {
            const uint32_t *p = w + 4u * u;
            const uint32_t e = p[4];
            v = make_uint4(funnel_r(p[0], p[1], sh), funnel_r(p[1], p[2], sh), funnel_r(p[2], p[3], sh),
                           funnel_r(p[3], e, sh));
        }
        __syncwarp();
        if (u < units) o[u] = v;
        __syncwarp();
    }
    warp_copy_ordered(dst, d + 16u * units, src, s + 16u * units, len & 15u, lane);
}

// Copy a match of ML bytes at distance off to dst[op..] (off <= op) by one warp.
BSG_D void dec_match(uint8_t *dst, uint32_t op, uint32_t off, uint32_t ML, uint32_t lane)
{
    if (off > 4u || off == 3u) {
        lz4_match_copy(dst, op, off, ML, lane);
        return;
    }
    // period 1, 2 or 4: every aligned word of the output is the same
    uint32_t p = ld32u(dst, op - off);
    if (off == 1u) p = (p & 0xffu) * 0x01010101u;
    if (off == 2u) p = (p & 0xffffu) * 0x00010001u;
    p = rotl(p, 8u * (op & 3u));             // byte 0 of p lies at op: the word at op & ~3
    const uint32_t end = op + ML;
    uint32_t a = (op + 3u) & ~3u, z = end & ~3u;
    __syncwarp();
    if (a > z) a = z = end;                  // within a word
    if (op + lane < a) dst[op + lane] = (uint8_t)(p >> (8u * ((op + lane) & 3u)));
    if (lane >= 4u && z + lane - 4u < end) dst[z + lane - 4u] = (uint8_t)(p >> (8u * (lane & 3u)));
    uint32_t *d32 = reinterpret_cast<uint32_t *>(dst);
    uint32_t i = (a >> 2) + lane, n = z >> 2;
    if (ML >= 512u) {
        // whole 16-byte units in the middle of a long run
        const uint32_t u0 = (a + 15u) >> 4, u1 = z >> 4;
        uint4 *d128 = reinterpret_cast<uint4 *>(dst);
#pragma unroll 1
        for (uint32_t u = u0 + lane; u < u1; u += 32) d128[u] = make_uint4(p, p, p, p);
        if (i < 4u * u0) d32[i] = p;
        i = 4u * u1 + lane;
    }
#pragma unroll 1
    for (; i < n; i += 32) d32[i] = p;
}

// Strict decode of the clen bytes src[ip0 ..] into exactly S bytes of dst by
// a CTA of 64 threads (src and dst word-aligned shared buffers, src readable 8
// bytes past the end; ring: DEC_RING_WORDS words of shared memory, 8-byte
// aligned).  dst is 16-byte aligned.  True when the block is valid; every
// thread returns the same after a barrier.  The rules are lz4_decode_warp's.
BSG_D bool cta_lz4_decode(const uint8_t *src, uint32_t ip0, uint32_t clen, uint8_t *dst, uint32_t S,
                          uint32_t *ring, uint32_t tid)
{
    const uint32_t lane = tid & 31u, end = ip0 + clen;
    const bool parser = tid < 32u;
    uint2 *seq = reinterpret_cast<uint2 *>(ring);
    uint32_t *ctl = ring + 4u * DEC_BATCH;
    uint32_t ip = ip0, op = 0;
    for (uint32_t step = 0;; step++) {
        const uint32_t half = (step & 1u) * DEC_BATCH;
        if (parser) {
            uint32_t n = 0, state = 0;   // 1: the block ends well, 2: it is corrupt
#pragma unroll 1
            for (; n < DEC_BATCH; n++) {
                // every pass consumes at least its token byte, so the loop ends
                state = 2;
                if (ip >= end) break;
                const uint32_t token = src[ip];
                uint32_t b = src[ip + 1];
                uint32_t LL = token >> 4;
                ip++;
                if (LL == 15u) {
                    if (b != 255u && ip < end) {
                        LL += b;
                        ip++;
                    } else if (!lz4_read_len(src, end, ip, LL, lane)) {
                        break;
                    }
                }
                if ((LL > end - ip) | (LL > S - op)) break;
                if (LL) dec_literals(dst, op, src, ip, LL, lane);
                ip += LL;
                op += LL;
                if (ip == end) {
                    state = op == S ? 1 : 2;
                    break;
                }
                if (end - ip < 2u) break;
                // (in place: the literals end before the input that follows)
                const uint32_t off = (uint32_t)src[ip] | ((uint32_t)src[ip + 1] << 8);
                b = src[ip + 2];
                ip += 2;
                uint32_t ML = token & 15u;
                if (ML == 15u) {
                    if (b != 255u && ip < end) {
                        ML += b;
                        ip++;
                    } else if (!lz4_read_len(src, end, ip, ML, lane)) {
                        break;
                    }
                }
                ML += LZ4_MINMATCH;
                // (ML is below 2^31: at most 255 per stream byte)
                // In place the match must not reach what the parser has still to
                // read either: by that margin only a corrupt block's would.
                const uint32_t last = S - LZ4_LASTLITERALS, room = src == dst && ip < last ? ip : last;
                if ((off == 0) | (off > op) | (op + ML > room) | (op + LZ4_MFLIMIT > S)) break;
                if (lane == 0) seq[half + n] = make_uint2(op | (off << 16), ML);
                op += ML;
                state = 0;
            }
            if (lane == 0) ctl[step & 1u] = n | (state << 8);
        } else if (step > 0) {
            const uint32_t n = ctl[(step & 1u) ^ 1u] & 255u;
#pragma unroll 1
            for (uint32_t k = 0; k < n; k++) {
                const uint2 m = seq[(half ^ DEC_BATCH) + k];
                dec_match(dst, m.x & 0xffffu, m.x >> 16, m.y, lane);
                __syncwarp();
            }
        }
        __syncthreads();
        const uint32_t c = ctl[step & 1u], state = c >> 8;
        if (state) {
            if (!parser && state == 1u) {
#pragma unroll 1
                for (uint32_t k = 0; k < (c & 255u); k++) {
                    const uint2 m = seq[half + k];
                    dec_match(dst, m.x & 0xffffu, m.x >> 16, m.y, lane);
                    __syncwarp();
                }
            }
            __syncthreads();
            return state == 1u;
        }
    }
}

#endif  // __CUDACC__ || BSG_WARP_EMU

}  // namespace bsg
