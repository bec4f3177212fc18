// CPU test of the CTA-wide device code of paper_1503_00638_gb300/csrc (the
// in-place bit transpose, the level-0 LZ4 encoder and the two-warp decoder)
// on the CTA emulator: the transpose against the oracle's, the encoder byte
// for byte against the one-warp encoder's parse (lz4_encode_bitmap, run on a
// CTA of one warp) and through the oracle's decoder, the decoder in place on
// both encoders' blocks and, for its verdict, on damaged ones.  argv: element size, elements, kind, seed.
#include "cta_emu.h"
#include "../../paper_1503_00638_gb300/csrc/lz4_cta.cuh"
#include "../../paper_1503_00638_gb300/csrc/lz4_cta_dec.cuh"
#include "../../paper_1503_00638_gb300/csrc/shuffle_cta.cuh"
#include <random>
extern "C" {
size_t orc_lz4_compress_block(const uint8_t *src, size_t n, uint8_t *dst, size_t cap);
int orc_lz4_decompress_block(const uint8_t *src, size_t src_len, uint8_t *dst, size_t dst_len);
int orc_bitshuffle(const void *vin, void *vout, size_t n, size_t es, size_t block_elems, int inverse);
}
using namespace bsg;
alignas(16) static uint8_t buf[65536 + 64], out[70000], ref[70000], scr[65536], bm[65536];

template <int ES> static void transpose(uint32_t Bb)
{
    uint32_t v[32];
    const uint32_t u = threadIdx.x, units = cta_units<ES>(Bb);
    if (u < units) cta_get_rows<ES>(buf, Bb, u, v, [](uint32_t, uint32_t (&)[32]) {});
    __syncthreads();
    if (u < units) cta_put_rows<ES>(buf, Bb, u, v);
    __syncthreads();
    if (!cta_rows_whole<ES>(Bb)) cta_pack_rows<ES>(buf, Bb);
}

// The block's image at phase `ph` near the end of the buffer, as the kernel
// places it, decoded to the buffer's start by two warps.
static bool decode_in_place(const uint8_t *img, uint32_t cs, uint32_t S, uint32_t ph)
{
    alignas(16) static uint8_t D[70000];
    alignas(16) static uint32_t ring[DEC_RING_WORDS];
    const uint32_t E = (S + 2u * S / 255u + 160u + 15u) & ~15u, off = (E - (cs + 4u) - 32u) & ~15u;
    memset(D, 0x5A, sizeof D);
    memcpy(D + off + ph + 4, img, cs);
    bool ok = false;
    run_cta(64, [&] {
        const bool r = cta_lz4_decode(D, off + ph + 4, cs, D, S, ring, threadIdx.x);
        if (threadIdx.x == 0) ok = r;
    });
    memcpy(buf, D, S);
    return ok;
}

int main(int argc, char **argv)
{
    if (argc < 5) return 2;
    const uint32_t es = (uint32_t)atoi(argv[1]), Bb = (uint32_t)atoi(argv[2]);
    const int kind = atoi(argv[3]);
    std::mt19937 rng((unsigned)atoi(argv[4]));
    const uint32_t S = Bb * es, W = cta_warps(S), rowlen = Bb / 8;
    std::vector<uint8_t> x(S), rows(S), back(S);
    if (kind == 0) {            // a random walk
        int64_t w = 0;
        for (uint32_t i = 0; i < Bb; i++) {
            w += (rng() & 1 ? 1 : -1) * (1 << (rng() % 7));
            memcpy(x.data() + (size_t)i * es, &w, es);
        }
    } else {                    // bit-rows of stretches: zeros, runs, copies of the row above, noise
        const uint32_t R = rowlen;
        uint32_t i = 0;
        while (i < S) {
            const int k = (int)(rng() % 6);
            uint32_t len = 1 + rng() % (kind == 1 ? 40 : kind == 2 ? 3000 : 9);
            if (kind == 3 && (k == 3 || k == 4)) len = 12;   // many short matches: the node tables overflow
            for (; len && i < S; len--, i++) {
                const uint8_t r = (uint8_t)rng();
                rows[i] = k == 0 ? 0 : k == 1 ? r : k == 2 ? (i >= R ? rows[i - R] : r)
                        : k == 3 ? (i >= 4 ? rows[i - 4] : r) : k == 4 ? (i >= R ? rows[i - R] : 0) : (r & 1);
            }
        }
        orc_bitshuffle(rows.data(), x.data(), Bb, es, Bb, 1);
    }
    orc_bitshuffle(x.data(), rows.data(), Bb, es, Bb, 0);
    memset(buf, 0xA5, sizeof buf);
    memcpy(buf, x.data(), S);
    memset(out, 0, sizeof out);
    memset(scr, 0x5A, sizeof scr);
    const uint32_t hbits = cta_hbits(S);
    if (cta_scratch_bytes<0>(W) > sizeof scr || cta_scratch_bytes<1>(W, hbits) > sizeof scr) return 3;
    uint32_t cs = 0, known = 0;
    uint8_t *enc = out + 4;   // the slot's four length bytes come first
    run_cta(32 * W, [&] {
        switch (es) {
        case 1: transpose<1>(Bb); break;
        case 2: transpose<2>(Bb); break;
        case 4: transpose<4>(Bb); break;
        default: transpose<8>(Bb); break;
        }
        const CtaScratch c = cta_scratch<0>(scr, W);
        cta_eq_bitmaps(reinterpret_cast<const uint32_t *>(buf), S / 4, (rowlen & 3u) ? 0u : rowlen / 4, c, W);
        __syncthreads();
        const uint32_t o = cta_lz4_encode<0>(buf, S, rowlen, enc, c, W, hbits, [&](uint32_t s) {
            if (threadIdx.x == 0) known = s;
        }, [] {});
        if (threadIdx.x == 0) cs = o;
    });
    if (memcmp(buf, rows.data(), S)) { fprintf(stderr, "transpose differs\n"); return 1; }
    uint32_t want = 0;
    run_cta(32, [&] {
        const uint32_t o = lz4_encode_bitmap(buf, S, rowlen, ref, reinterpret_cast<uint32_t *>(bm));
        if (threadIdx.x == 0) want = o;
    });
    if (cs != want || known != cs || cs > lz4_bound(S) || memcmp(enc, ref, cs)) {
        uint32_t k = 0;
        while (k < cs && enc[k] == ref[k]) k++;
        fprintf(stderr, "encoding differs: %u / %u bytes, known %u, first at %u\n", cs, want, known, k);
        return 1;
    }
    if (orc_lz4_decompress_block(enc, cs, back.data(), S) || memcmp(back.data(), rows.data(), S)) {
        fprintf(stderr, "the oracle rejects the block\n");
        return 1;
    }
    // level 1 against the one-warp encoder's search and emission
    alignas(16) static uint8_t out1[70000];
    uint32_t cs1 = 0;
    const uint32_t W1 = (S + 8191) / 8192;
    run_cta(32 * W1, [&] {
        const CtaScratch c = cta_scratch<1>(scr, W1, hbits);
        const uint32_t o = cta_lz4_encode<1>(buf, S, rowlen, out1 + 4, c, W1, hbits, [](uint32_t) {}, [] {});
        if (threadIdx.x == 0) cs1 = o;
    });
    run_cta(32, [&] {
        const uint32_t o = hbits == 11   ? lz4_encode_warp<1, 11>(buf, S, rowlen, ref, (uint16_t *)bm)
                           : hbits == 12 ? lz4_encode_warp<1, 12>(buf, S, rowlen, ref, (uint16_t *)bm)
                                         : lz4_encode_warp<1, 13>(buf, S, rowlen, ref, (uint16_t *)bm);
        if (threadIdx.x == 0) want = o;
    });
    if (cs1 != want || memcmp(out1 + 4, ref, cs1)) {
        fprintf(stderr, "level 1 differs: %u / %u bytes\n", cs1, want);
        return 1;
    }
    std::vector<uint8_t> oc(lz4_bound(S) + 16);
    const uint32_t ocs = (uint32_t)orc_lz4_compress_block(rows.data(), S, oc.data(), oc.size());
    for (int who = kind & 1; who < 2; who++)   // (the CTA's threads are real ones: slow)
        for (uint32_t ph : {who ? 5u : 15u})
            if (!decode_in_place(who ? oc.data() : enc, who ? ocs : cs, S, ph) || memcmp(buf, rows.data(), S)) {
                fprintf(stderr, "decoding in place differs, phase %u, encoder %d\n", ph, who);
                return 1;
            }
    // a byte changed, the end cut off: the verdict of the oracle's decoder
    for (int t = 0; t < (S <= 4096 && kind < 2 ? 3 : 0); t++) {
        std::vector<uint8_t> bad(oc.begin(), oc.begin() + ocs);
        if (t % 3 == 2)
            bad.resize(rng() % bad.size());
        else
            bad[rng() % bad.size()] = (uint8_t)rng();
        const bool want_ok = !bad.empty() && orc_lz4_decompress_block(bad.data(), bad.size(), back.data(), S) == 0;
        std::vector<uint8_t> img(bad);
        img.resize(bad.size() + 16, 0xEE);
        if (decode_in_place(img.data(), (uint32_t)bad.size(), S, 3) != want_ok) {
            fprintf(stderr, "verdict on a damaged block differs (%d)\n", t);
            return 1;
        }
    }
    printf("ok %u -> %u\n", S, cs);
    return 0;
}
