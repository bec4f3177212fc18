// The decompress kernel of blocks over 8 KiB: LZ4 decode in place -> bit
// un-transpose (Sec. 4.2.1), a CTA of two warps per block.
#pragma once

#include "codec.cuh"
#include "lz4_cta_dec.cuh"
#include "shuffle.cuh"

namespace bsg {

// Buffer for decoding blocks of S bytes in place: room for the image (4 +
// lz4b(S), placed at most 48 bytes before the end) and the margin of
// decompress_inplace_kernel's argument (S + 2 S / 255 + 49).
__host__ __device__ constexpr uint32_t dec_cta_buf(uint32_t S) { return r16(S + 2u * S / 255u + 160u); }
static_assert(dec_cta_buf(8) >= 4 + lz4b(8) + 48 && dec_cta_buf(8192) >= 4 + lz4b(8192) + 48 &&
                  dec_cta_buf(65536) >= 4 + lz4b(65536) + 48 &&
                  dec_cta_buf(65536) >= 65536 + 2 * 65536 / 255 + 49,
              "in-place buffer");

__host__ __device__ constexpr uint32_t dec_cta_smem(uint32_t S)
{
    return dec_cta_buf(S) + r16(4u * DEC_RING_WORDS) + 32u;
}

// The 12-byte header of the stream (one warp).
BSG_D void dec_check_header(const CodecArgs &a, uint32_t lane)
{
    uint32_t ok = 1;
    if (lane < 12) {
        const uint8_t want = lane < 8 ? (uint8_t)((a.n_elem * a.es) >> (8 * (7 - lane)))
                                      : (uint8_t)(((uint64_t)a.B * a.es) >> (8 * (11 - lane)));
        ok = a.in_bytes >= 12 && a.in[lane] == want;
    }
    if (__ballot_sync(FULL, !ok) && lane == 0) set_status(a.status, BSGPU_ERR_CORRUPT);
}

// Persistent, one buffer per CTA: the first warp fetches a block's bytes to the
// buffer's end (one bulk copy and the ragged edges) and parses, the second
// copies the matches (cta_lz4_decode); both un-transpose, from the bit-rows
// straight to the output.
//
// Shared memory holds 12, 6 or 3 blocks of 16, 32 or 64 KiB per SM: with a warp
// each the chain of tokens leaves the SM idle.  201 MB of int32 in blocks of
// 16, 32 and 64 KiB: 164, 258 and 424 us with one warp per block, 155, 212 and
// 334 us with two.  Blocks of at most 8 KiB keep one warp (the in-place kernel
// of kernels.cu): there 20 parsing warps per SM are issue-bound, and two warps
// a block, 16 blocks per SM, took 1.25 to 1.6 times as long.  8-byte
// elements keep one warp up to 16 KiB too, and have 96 registers above (with 80
// their un-transpose spilled: 67 MB in 32 KiB blocks 69 -> 65 us).
template <int ES>
__global__ void __launch_bounds__(64, ES == 8 ? 10 : 12) decompress_cta_kernel(const __grid_constant__ CodecArgs a)
{
    extern __shared__ __align__(128) uint8_t sm[];
    const uint32_t BUF = dec_cta_buf(a.B * ES);
    uint8_t *buf = sm;
    uint32_t *ring = reinterpret_cast<uint32_t *>(sm + BUF);
    uint32_t *next = ring + DEC_RING_WORDS;
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + dec_cta_smem(a.B * ES) - 16u);
    const uint32_t tid = threadIdx.x, lane = tid & 31u;
    const bool first_warp = tid < 32u;
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
        *next = atomicAdd(a.tile_counter, 1u);
    }
    __syncthreads();
    uint32_t tile = *next, parity = 0;
    __syncthreads();
    DecLoad ld{};
    if (first_warp) {
        if (blockIdx.x == 0) dec_check_header(a, lane);
        if (tile < a.nb) ld = dec_issue(a, tile, buf, bar, lane, BUF);
    }
    while (tile < a.nb) {
        uint32_t ip0 = 0, clen = 0;   // (an empty image fails to decode)
        if (first_warp) {
            if (lane == 0) *next = atomicAdd(a.tile_counter, 1u);
            if (ld.bulk) {
                if (!mbar_wait_bounded(bar, parity) && lane == 0) set_status(a.status, BSGPU_ERR_TIMEOUT);
                parity ^= 1u;
            }
            if (ld.ok) {
                uint8_t *comp = buf + ld.off;
                if (ld.eidx != ~0u) comp[ld.eidx] = ld.ebyte;
                __syncwarp();
                if (get_be32(comp + ld.delta) == ld.clen) {
                    ip0 = ld.off + ld.delta + 4u;
                    clen = ld.clen;
                }
            }
        }
        const uint32_t Bb = block_elems_of(a, tile), S = Bb * ES;
        const bool good = cta_lz4_decode(buf, ip0, clen, buf, S, ring, tid);
        const uint32_t nxt = *next;
        if (!good && tid == 0) set_status(a.status, BSGPU_ERR_CORRUPT);
        uint8_t *dst = a.out + (uint64_t)tile * a.B * ES;
        if (good) unshuffle_block(buf, dst, Bb, ES, tid, 64);
        if (tile + 1 == a.nb) {
            const uint32_t tb = a.tail_elems * ES;
            const uint64_t first = (a.n_elem - a.tail_elems) * ES;
            if (a.in_bytes >= tb && tid < tb) a.out[first + tid] = a.in[a.in_bytes - tb + tid];
        }
        // the buffer's generic accesses before the next fetch
        fence_proxy_async_smem();
        __syncthreads();
        if (first_warp) {
            ld = DecLoad{};
            if (nxt < a.nb) ld = dec_issue(a, nxt, buf, bar, lane, BUF);
        }
        tile = nxt;
    }
}

template <int ES>
cudaError_t launch_decompress_cta_es(const CodecArgs &a, cudaStream_t s)
{
    auto kernel = decompress_cta_kernel<ES>;
    const uint32_t smem = dec_cta_smem(a.B * ES);
    const cudaError_t e = allow_smem(kernel, smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 148, per = 1;
    if (cudaGetDevice(&dev) == cudaSuccess)
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, 64, smem) != cudaSuccess || per < 1)
        per = 1;
    uint64_t grid = (uint64_t)sms * (uint32_t)per;
    if (grid > a.nb) grid = a.nb;
    kernel<<<(uint32_t)grid, 64, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace bsg
