// CPU test of the CTA's level-0 encoder around the number of parse-graph nodes
// that its tables hold: blocks of exactly so many runs of equal words, one
// fewer and more, up to as many as fit, against the one-warp encoder byte for
// byte.  argv: block bytes, nodes (0: the usual number).
#include "cta_emu.h"
#include "../../paper_1503_00638_gb300/csrc/lz4_cta.cuh"
#include <random>
extern "C" int orc_lz4_decompress_block(const uint8_t *src, size_t src_len, uint8_t *dst, size_t dst_len);
using namespace bsg;
alignas(16) static uint8_t buf[65536 + 64], out[70000], ref[70000], scr[65536], bm[65536], back[65536];

int main(int argc, char **argv)
{
    if (argc < 3) return 2;
    const uint32_t S = (uint32_t)atoi(argv[1]), NW = S / 4, W = cta_warps(S), rowlen = S / 32;
    const uint32_t cap = atoi(argv[2]) ? (uint32_t)atoi(argv[2]) : cta_node_cap(W), most = NW / 5;
    std::mt19937 rng(S);
    uint32_t *w = reinterpret_cast<uint32_t *>(buf);
    for (uint32_t K : {0u, 1u, cap - 2, cap - 1, cap, cap + 1, most}) {
        if (K > most) continue;
        for (uint32_t i = 0; i < NW; i++) w[i] = rng();
        for (uint32_t k = 0; k < K; k++)   // a word four times: one run of candidates
            for (uint32_t j = 2; j < 5; j++) w[5 * k + j] = w[5 * k + 1];
        memset(scr, 0x5A, sizeof scr);
        uint32_t cs = 0, want = 0;
        run_cta(32 * W, [&] {
            const CtaScratch c = cta_scratch<0>(scr, W, 0, cap);
            cta_eq_bitmaps<1>(w, NW, rowlen / 4, c, W);
            __syncthreads();
            const uint32_t o = cta_lz4_encode<0>(buf, S, rowlen, out + 4, c, W, 0, [](uint32_t) {}, [] {});
            if (threadIdx.x == 0) cs = o;
        });
        run_cta(32, [&] {
            const uint32_t o = lz4_encode_bitmap(buf, S, rowlen, ref, reinterpret_cast<uint32_t *>(bm));
            if (threadIdx.x == 0) want = o;
        });
        if (cs != want || memcmp(out + 4, ref, cs) || cta_scratch_bytes<0>(W, 0, cap) > sizeof scr ||
            orc_lz4_decompress_block(out + 4, cs, back, S) || memcmp(back, buf, S)) {
            fprintf(stderr, "%u runs, tables of %u: %u / %u bytes\n", K, cap, cs, want);
            return 1;
        }
        // nothing past the scratch that the plan reserves
        for (size_t k = cta_scratch_bytes<0>(W, 0, cap); k < sizeof scr; k++)
            if (scr[k] != 0x5A) {
                fprintf(stderr, "%u runs: scratch written past its end\n", K);
                return 1;
            }
    }
    printf("ok\n");
    return 0;
}
