// CPU test of the in-place LZ4 decoders on corrupt blocks whose output passes
// the input that is still to be read (a long early match, more input behind
// it than a valid block can have): they must give the oracle's verdict and
// must not write over unread input.  argv: block bytes, phase of the image.
#include "cta_emu.h"
#include "../../paper_1503_00638_gb300/csrc/lz4_cta_dec.cuh"
extern "C" int orc_lz4_decompress_block(const uint8_t *src, size_t src_len, uint8_t *dst, size_t dst_len);
using namespace bsg;

static void put_len(std::vector<uint8_t> &b, uint32_t v)
{
    for (v -= 15; v >= 255; v -= 255) b.push_back(255);
    b.push_back((uint8_t)v);
}

// One literal, a match of distance 1 that ends at output byte `to`, then
// four-byte matches (each brings the output a byte nearer to the input) up to
// `shorts`, then bytes `pad` up to clen.
static std::vector<uint8_t> block(uint32_t to, uint32_t shorts, uint8_t pad, uint32_t clen)
{
    std::vector<uint8_t> b{0x1f, 0x10, 1, 0};
    put_len(b, to - 1 - LZ4_MINMATCH);
    for (uint32_t k = 0; k < shorts; k++) b.insert(b.end(), {0x00, 1, 0});
    b.resize(clen, pad);
    return b;
}

int main(int argc, char **argv)
{
    if (argc < 3) return 2;
    const uint32_t S = (uint32_t)atoi(argv[1]), ph = (uint32_t)atoi(argv[2]);
    alignas(16) static uint8_t D[70000], back[70000];
    alignas(16) static uint32_t ring[DEC_RING_WORDS];
    const uint32_t clen = S + S / 255 - 8;
    const uint32_t E = (S + 2u * S / 255u + 160u + 15u) & ~15u, off = (E - (clen + 4u) - 32u) & ~15u;
    const uint32_t ip0 = off + ph + 4;
    // how far behind the input the long match ends (negative: past it)
    for (int d : {-(int)(S / 2), -1, 0, 1, 13, 14, 15, 30})
        for (uint8_t pad : {0x00, 0x10, 0xf0, 0xff}) {
            // the match ends at ip - d; its length bytes are part of ip
            uint32_t to = ip0 + 4u - (uint32_t)d, ext = 0;
            while ((to - 5u - 15u) / 255u + 1u != ext) {
                ext = (to - 5u - 15u) / 255u + 1u;
                to = ip0 + 4u + ext - (uint32_t)d;
            }
            const std::vector<uint8_t> img = block(to, 40, pad, clen);
            // the sequence that first takes the output past the input is never applied
            const uint32_t read = 4u + ext + (d < 0 ? 0u : 3u * ((uint32_t)d + 1u));
            const bool want = orc_lz4_decompress_block(img.data(), clen, back, S) == 0;
            for (int warps : {1, 2}) {
                memset(D, 0x5A, sizeof D);
                memcpy(D + ip0, img.data(), clen);
                bool ok = false;
                run_cta(32 * warps, [&] {
                    const bool r = warps == 2 ? cta_lz4_decode(D, ip0, clen, D, S, ring, threadIdx.x)
                                              : lz4_decode_warp<true>(D + off, ph + 4, clen, D, S) == 0;
                    if (threadIdx.x == 0) ok = r;
                });
                const bool whole = memcmp(D + ip0 + read, img.data() + read, clen - read) == 0;
                if (want || ok || !whole) {
                    fprintf(stderr, "%d warps, match %d bytes behind the input, padding %02x: verdict %d, oracle %d, unread input %s\n",
                            warps, d, pad, ok, want, whole ? "whole" : "overwritten");
                    return 1;
                }
            }
        }
    printf("ok\n");
    return 0;
}
