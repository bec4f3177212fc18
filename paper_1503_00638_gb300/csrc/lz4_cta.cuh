// LZ4 block encoder for a CTA of W warps (Sec. 4.1, 4.2.1), for blocks of up to
// 64 KiB: at level 0 the same greedy parse, byte for byte, as
// lz4_encode_bitmap and lz4_encode_bitmap_fast (lz4_warp.cuh has the format
// and the parse graph), at level 1 that of lz4_encode_warp.
//
// Why a CTA and not a warp: the block is the unit that shared memory holds,
// so one warp per block leaves an SM with as many warps as blocks fit (20 at
// 8 KiB, 3 at 64 KiB) and the encoder bound by the latency of one warp's
// serial steps.  Here a block of S bytes gets a thread per 128 bytes: 28 to 32
// warps per SM for every block size, each thread holding one 32-word group of
// the bit transpose.
//
// The stages of level 0, a barrier between each:
//   1. word-equality bitmaps E[k] = {row, run} (the caller, or
//      cta_eq_bitmaps from shared memory);
//   2. thread u derives the candidates of bitmap word u, their run ends and,
//      by a scan, the ranks of the run ends (the parse graph's nodes);
//   3. the nodes' positions, then each node's successor;
//   4. warp 0 walks the graph by pointer jumping and leaves up to one
//      sequence descriptor per thread;
//   5. each thread places its sequence by a scan of the sizes and writes its
//      token, lengths, offset and the ragged ends of its literal run;
//   6. the 16-byte units of all literal runs form one list that the warps
//      copy 32 units at a time, whatever the lengths of the single runs
//      (copying run by run, four at a time, kept many lanes idle: it was the
//      largest part of the one-warp encoder's instructions; a list of 4-byte
//      words still took 1140 of a CHIME-shaped block's 5070 warp
//      instructions).
// At level 1 the search is a chain (where it probes depends on what it found):
// the first warp searches (lz4_next_match) for a descriptor per thread, then
// stages 5 and 6 write those sequences, instead of one sequence after another
// by the warp that searches.
#pragma once

#include "lz4_warp.cuh"

namespace bsg {

#if defined(__CUDACC__) || defined(BSG_WARP_EMU)

// The thread's index, read anew: what is computed from it is not carried
// through the persistent loop in registers (the compiler otherwise hoists
// every per-thread address out of the loop and spills them).
BSG_D uint32_t fresh_tid()
{
#ifdef BSG_WARP_EMU
    return threadIdx.x;
#else
    uint32_t t;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
    return t;
#endif
}

// Warps for a block of S bytes: one thread per 128 bytes.
__host__ __device__ constexpr uint32_t cta_warps(uint32_t S) { return (S + 4095u) / 4096u; }

// Nodes of the parse graph that the tables hold for W warps' blocks unless the
// caller gives more room; a block with more walks from candidate to match end
// (the same bytes).  The CHIME-shaped data has 32 nodes per 8 KiB block on
// average, 80 at most.
__host__ __device__ constexpr uint32_t cta_node_cap(uint32_t W) { return 64u * W; }
// Words of the bitmaps and, over them, of the four jump tables.
__host__ __device__ constexpr uint32_t cta_bitmap_words(uint32_t W, uint32_t cap)
{
    const uint32_t maps = 2u * (32u * W + 1u) + 5u * 32u * W, jumps = 2u * cap;
    return maps > jumps ? maps : jumps;
}

constexpr uint32_t CTA_MAX_WARPS = 16;   // 64 KiB blocks
constexpr uint32_t CTA_NONE = 0xffffu;

// Shared scratch of W warps, in 32-bit words.
struct CtaScratch {
    uint2 *E;         // 32 W + 1 equality bitmap words {row, run}
    uint32_t *cer;    // run-end bitmaps of bit-row and of run candidates
    uint32_t *ceu;
    uint32_t *any;    // candidates of either kind
    uint32_t *row;    // bit-row candidates
    uint32_t *pre;    // run ends before a bitmap word: bit-row | run << 16
    uint2 *node;      // {position, first candidate | successor << 16}
    uint2 *desc;      // sequences {match start | offset << 16, match end}, then the
                      // literal list's entries
    uint32_t *ex;     // exchange words between the warps (EX_*)
    uint16_t *table;  // level 1: the hash table (2^hbits entries), the rest but
                      // desc and ex unused
    uint16_t *jmp;    // jump tables: over E to pre, dead by then
    uint32_t cap;     // nodes the tables hold, 0 for cta_node_cap(W)
};
enum : uint32_t { EX_NZ = 0, EX_CNT = 16, EX_SCAN = 32, EX_LIT = 48, EX_CTL = 64, EX_WORDS = 72 };

// Hash bits of level 1 for blocks of S bytes.
__host__ __device__ constexpr uint32_t cta_hbits(uint32_t S) { return S <= 8192u ? 11u : S <= 16384u ? 12u : 13u; }

// (level 0: with tables of `cap` nodes, 0 for cta_node_cap(W))
template <int LEVEL>
__host__ __device__ constexpr uint32_t cta_scratch_bytes(uint32_t W, uint32_t hbits = 0, uint32_t cap = 0)
{
    return LEVEL >= 1 ? (2u << hbits) + 4u * (2u * (32u * W + 1u) + EX_WORDS)
                      : 4u * ((cap ? cta_bitmap_words(W, cap) + 2u * cap
                                   : 2u * (32u * W + 1u) + 5u * 32u * W + 2u * cta_node_cap(W)) +
                              2u * (32u * W + 1u) + EX_WORDS);
}

template <int LEVEL>
BSG_D CtaScratch cta_scratch(uint8_t *base, uint32_t W, uint32_t hbits = 0, uint32_t cap = 0)
{
    CtaScratch c{};
    uint32_t *p = reinterpret_cast<uint32_t *>(base);   // 16-byte aligned
    if (LEVEL >= 1) {
        c.table = reinterpret_cast<uint16_t *>(p);
        p += (2u << hbits) / 4u;
    } else {
        uint32_t *const end = p + (cap ? cta_bitmap_words(W, cap) : 0u);
        c.cap = cap;
        c.E = reinterpret_cast<uint2 *>(p);
        c.jmp = reinterpret_cast<uint16_t *>(p);
        p += 2u * (32u * W + 1u);
        c.cer = p;
        c.ceu = p + 32u * W;
        c.any = p + 64u * W;
        c.row = p + 96u * W;
        c.pre = p + 128u * W;
        p += 160u * W;
        if (cap) p = end;
        c.node = reinterpret_cast<uint2 *>(p);
        p += 2u * (cap ? cap : cta_node_cap(W));
    }
    c.desc = reinterpret_cast<uint2 *>(p);
    p += 2u * (32u * W + 1u);
    c.ex = p;
    return c;
}

// the four jump tables fit the space of the bitmaps they replace
static_assert(4u * cta_node_cap(1) * 2u <= 4u * (2u * 33u + 64u), "jump tables");

// Equality bitmaps of the NW words at s32 from shared memory: E[k].x bit l
// set when word w = 32 k + l equals word w - R (R = 0: none), E[k].y when it
// equals word w - 1.  Followed by a barrier.  (UNROLL 8 where the number of words
// is known: 64 MiB of bytes in 8 KiB blocks 92 -> 88 us, of 16-bit samples 91 ->
// 87.)
template <int UNROLL = 1>
BSG_D void cta_eq_bitmaps(const uint32_t *s32, uint32_t NW, uint32_t R, const CtaScratch &c,
                          uint32_t W)
{
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t NB = (NW + 31u) / 32u;
#pragma unroll UNROLL
    for (uint32_t k = warp; k < NB; k += W) {
        const uint32_t w = 32u * k + lane;
        const bool in = w < NW;
        const uint32_t x = in ? s32[w] : 0u;
        const uint32_t xp = in && w > 0 ? s32[w - 1u] : ~x;
        const uint32_t xr = in && R && w >= R ? s32[w - R] : ~x;
        const uint32_t row = __ballot_sync(FULL, in && x == xr);
        const uint32_t run = __ballot_sync(FULL, in && x == xp);
        if (lane == 0) c.E[k] = make_uint2(row, run);
    }
}

// First candidate in [from, to], ~0u when none: the bitmap words and, past an
// empty one, the warps' masks of non-zero words.
BSG_D uint32_t cta_first_set(const CtaScratch &c, uint32_t from, uint32_t to, uint32_t W)
{
    if (from > to) return ~0u;
    uint32_t k = from >> 5;
    uint32_t m = c.any[k] & (~0u << (from & 31u));
    if (m == 0) {
        k++;
        uint32_t j = k >> 5;
        if (j >= W) return ~0u;
        uint32_t z = c.ex[EX_NZ + j] & (~0u << (k & 31u));
        while (z == 0) {
            if (++j >= W) return ~0u;
            z = c.ex[EX_NZ + j];
        }
        k = 32u * j + (uint32_t)(__ffs(z) - 1);
        m = c.any[k];
    }
    const uint32_t w = 32u * k + (uint32_t)(__ffs(m) - 1);
    return w <= to ? w : ~0u;
}

// Encode src[0, S) (shared, word aligned, readable to S + 8; S a multiple of
// 8, at most 4096 W at level 0 and 8192 W at level 1) into dst (4 bytes past a 16-byte boundary, capacity
// lz4_bound(S)); c.E
// holds the block's bitmaps, a barrier passed since they were written.
// size_known(cs) is called by every thread as soon as the size is known,
// before the literal runs are copied; idle() once by the last warp, when
// there is more than one, while the first alone walks the parse graph.
// Returns the size; the caller's next barrier ends the reads of src.
// (Level 1: c.E is not used; hbits as cta_hbits of the stream's full blocks.)
template <int LEVEL, class SizeKnown, class Idle>
BSG_D uint32_t cta_lz4_encode(const uint8_t *src, uint32_t S, uint32_t rowlen, uint8_t *dst,
                              const CtaScratch &c, uint32_t W, uint32_t hbits, SizeKnown size_known,
                              Idle idle)
{
    const uint32_t tid = fresh_tid(), lane = tid & 31u, warp = tid >> 5, NT = 32u * W;
    const uint32_t *s32 = reinterpret_cast<const uint32_t *>(src);
    const uint32_t NB = (S / 4u + 31u) / 32u;
    const uint32_t R = (rowlen & 3u) ? 0u : rowlen / 4u;
    const uint32_t cap_nodes = c.cap ? c.cap : cta_node_cap(W);

    const bool some = LEVEL >= 1 || (S >= LZ4_MFLIMIT + 1u && S >= LZ4_LASTLITERALS + LZ4_L0_MINMATCH);
    const uint32_t wlim = some ? (S - LZ4_LASTLITERALS - LZ4_L0_MINMATCH) / 4u : 0u;
    const uint32_t matchlimit = S - LZ4_LASTLITERALS, cap = matchlimit / 4u;
    uint32_t N = 0, Nr = 0;   // nodes of the parse graph, those of the bit-row kind first
    bool graph = false;
    Lz4Probe probe;
    if (LEVEL >= 1) {
        uint4 *t4 = reinterpret_cast<uint4 *>(c.table);
        for (uint32_t i = tid; i < (2u << hbits) / 16u; i += NT) t4[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
    } else {
        // candidates: bits w, w + 1 and w + 2 set; a run of candidates ends where
        // the next bit is no candidate
        uint32_t cer = 0, ceu = 0, nz;
        {
            uint32_t crow = 0, crun = 0;
            if (tid < NB) {
                static_assert(LZ4_L0_MINWORDS == 3, "candidate masks");
                const uint2 e = c.E[tid], n = tid + 1u < NB ? c.E[tid + 1u] : make_uint2(0u, 0u);
                crow = e.x & funnel_r(e.x, n.x, 1u) & funnel_r(e.x, n.x, 2u);
                crun = e.y & funnel_r(e.y, n.y, 1u) & funnel_r(e.y, n.y, 2u);
                cer = crow & ~funnel_r(crow, (n.x & 7u) == 7u ? 1u : 0u, 1u);
                ceu = crun & ~funnel_r(crun, (n.y & 7u) == 7u ? 1u : 0u, 1u);
            }
            c.cer[tid] = cer;
            c.ceu[tid] = ceu;
            c.any[tid] = crow | crun;
            c.row[tid] = crow;
            nz = __ballot_sync(FULL, (crow | crun) != 0u);
        }
        const uint32_t cnt = (uint32_t)__popc(cer) | ((uint32_t)__popc(ceu) << 16);
        uint32_t incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(FULL, incl, d);
            if (lane >= (uint32_t)d) incl += t;
        }
        if (lane == 31) {
            c.ex[EX_NZ + warp] = nz;
            c.ex[EX_CNT + warp] = incl;
        }
        __syncthreads();
        uint32_t tot = 0, rank = incl - cnt;
#pragma unroll 1
        for (uint32_t j = 0; j < W; j++) {
            const uint32_t t = c.ex[EX_CNT + j];
            if (j < warp) rank += t;
            tot += t;
        }
        Nr = tot & 0xffffu;
        N = Nr + (tot >> 16);
        graph = some && N < cap_nodes;   // nodes 0 .. N - 1 and the start, N
        if (graph) {
            // node ids in position order within each kind, bit-row kind first
            c.pre[tid] = rank;
            uint32_t id = rank & 0xffffu;
#pragma unroll 1
            for (uint32_t m = cer; m; m &= m - 1u) c.node[id++].x = 32u * tid + (uint32_t)(__ffs(m) - 1);
            id = Nr + (rank >> 16);
#pragma unroll 1
            for (uint32_t m = ceu; m; m &= m - 1u) c.node[id++].x = 32u * tid + (uint32_t)(__ffs(m) - 1);
        }
        __syncthreads();
        if (graph) {
#pragma unroll 1
            for (uint32_t id = tid; id <= N; id += NT) {
                uint32_t p = 0;
                if (id < N) {
                    uint32_t e = c.node[id].x + LZ4_L0_MINWORDS;
                    if (e > cap) e = cap;
                    p = 4u * e;
                    if (p < matchlimit) {
                        const uint32_t x = s32[e] ^ s32[e - (id < Nr ? R : 1u)];
                        uint32_t eq = x ? ((uint32_t)(__ffs(x) - 1) >> 3) : 4u;
                        if (eq > matchlimit - p) eq = matchlimit - p;
                        p += eq;
                    }
                }
                const uint32_t w = cta_first_set(c, (p + 3u) / 4u, wlim, W);
                uint32_t succ = CTA_NONE << 16;
                if (w != ~0u) {
                    // the previous bit-row wins a tie
                    const uint32_t wd = w >> 5, below = (1u << (w & 31u)) - 1u;
                    const bool row = (c.row[wd] >> (w & 31u)) & 1u;
                    const uint32_t nx = row ? (c.pre[wd] & 0xffffu) + (uint32_t)__popc(c.cer[wd] & below)
                                            : Nr + (c.pre[wd] >> 16) + (uint32_t)__popc(c.ceu[wd] & below);
                    succ = w | (nx << 16);
                }
                c.node[id] = make_uint2(p, succ);
            }
        }
        __syncthreads();
    }
    uint32_t x0 = N, pos = 0;   // warp 0: where the next descriptors start
    bool more = some;
    if (W > 1 && warp == W - 1u) idle();
    if (graph && warp == 0) {
        // jmp[b * cap_nodes + x]: the node 2^(b + 1) steps after node x
#pragma unroll 1
        for (uint32_t x = lane; x <= N; x += 32) {
            const uint32_t y = c.node[x].y >> 16;
            c.jmp[x] = (uint16_t)(y == CTA_NONE ? CTA_NONE : c.node[y].y >> 16);
        }
        __syncwarp();
#pragma unroll 1
        for (uint32_t b = 1; b < 4; b++) {
            const uint16_t *jp = c.jmp + (b - 1u) * cap_nodes;
#pragma unroll 1
            for (uint32_t x = lane; x <= N; x += 32) {
                const uint32_t y = jp[x];
                c.jmp[b * cap_nodes + x] = y == CTA_NONE ? (uint16_t)CTA_NONE : jp[y];
            }
            __syncwarp();
        }
    }

    uint32_t o = 0, carry = 0;   // output written, end of the last match
    for (;;) {
        if (warp == 0) {
            uint32_t n = 0;
            if (LEVEL >= 1) {
#pragma unroll 1
                for (; more && n < NT; n++) {
                    uint32_t mp, off, len;
                    more = lz4_next_match<1>(src, S, rowlen, c.table, hbits, probe, lane, mp, off, len);
                    if (!more) break;
                    if (lane == 0) c.desc[n] = make_uint2(mp | (off << 16), mp + len);
                }
            } else if (graph) {
#pragma unroll 1
                while (more && n < NT) {
                    // lane k: the node k steps after x0 and the node after it
                    uint32_t x = x0;
                    if (lane & 1u) x = c.node[x].y >> 16;
#pragma unroll
                    for (uint32_t b = 0; b < 4; b++)
                        if (((lane >> (b + 1u)) & 1u) && x != CTA_NONE) x = c.jmp[b * cap_nodes + x];
                    const uint32_t succ = x != CTA_NONE ? c.node[x].y : CTA_NONE << 16;
                    const uint32_t nx = succ >> 16;
                    if (nx != CTA_NONE)
                        c.desc[n + lane] =
                            make_uint2(4u * (succ & 0xffffu) | ((nx < Nr ? rowlen : 4u) << 16), c.node[nx].x);
                    const uint32_t got = (uint32_t)__popc(__ballot_sync(FULL, nx != CTA_NONE));
                    x0 = __shfl_sync(FULL, nx, 31);
                    n += got;
                    more = got == 32u && x0 != CTA_NONE;
                }
            } else {
                for (; more && n < NT; n++) {
                    const uint32_t w = cta_first_set(c, (pos + 3u) / 4u, wlim, W);
                    if (w == ~0u) {
                        more = false;
                        break;
                    }
                    const bool row = (c.row[w >> 5] >> (w & 31u)) & 1u;
                    const uint32_t *ce = row ? c.cer : c.ceu;
                    // the candidate run holding w ends at or after it
                    uint32_t wd = w >> 5, m = ce[wd] & (~0u << (w & 31u));
                    while (m == 0 && wd + 1u < NT) m = ce[++wd];
                    uint32_t e = m ? 32u * wd + (uint32_t)(__ffs(m) - 1) + LZ4_L0_MINWORDS : cap;
                    if (e > cap) e = cap;
                    pos = 4u * e;
                    if (pos < matchlimit) {
                        const uint32_t x = s32[e] ^ s32[e - (row ? R : 1u)];
                        uint32_t eq = x ? ((uint32_t)(__ffs(x) - 1) >> 3) : 4u;
                        if (eq > matchlimit - pos) eq = matchlimit - pos;
                        pos += eq;
                    }
                    if (lane == 0) c.desc[n] = make_uint2(4u * w | ((row ? rowlen : 4u) << 16), pos);
                }
            }
            if (lane == 0) {
                c.ex[EX_CTL] = n;
                c.ex[EX_CTL + 1] = more ? 1u : 0u;
            }
        }
        __syncthreads();
        const uint32_t n = c.ex[EX_CTL];
        // the last literals take a thread of their own after the last sequence
        const bool fin = c.ex[EX_CTL + 1] == 0u && n < NT;
        const bool busy = 32u * warp <= n;   // warps past the last sequence only take part in the sums
        const bool mine = tid < n, last = fin && tid == n;
        uint32_t anchor = 0, mp = 0, ML = 0, off = 0, LL = 0, nll = 0, nml = 0, bytes = 0, units = 0;
        uint32_t sc = 0, lits = 0, packed = 0;
        if (busy) {
            anchor = tid == 0 ? carry : tid <= n ? c.desc[tid - 1u].y : 0u;
            mp = last ? S : anchor;
            if (mine) {
                const uint2 q = c.desc[tid];
                off = q.x >> 16;
                mp = q.x & 0xffffu;
                // back up over up to 3 equal bytes (never before the literal anchor)
                if (LEVEL == 0 && mp > anchor && mp > off) {
                    const uint32_t x = ld32u(src, mp - 4u) ^ ld32u(src, mp - 4u - off);
                    uint32_t back = (x ? (uint32_t)__clz(x) : 32u) >> 3;
                    if (back > 3u) back = 3u;
                    if (back > mp - anchor) back = mp - anchor;
                    if (back > mp - off) back = mp - off;
                    mp -= back;
                }
                ML = q.y - mp - LZ4_MINMATCH;
            }
            LL = mp - anchor;
            nll = lz4_ext_count(LL);
            nml = lz4_ext_count(ML);
            bytes = mine ? 3u + nll + LL + nml : last ? 1u + nll + LL : 0u;
            // one scan for both the output bytes (17 bits) and the entry's units
            // in the literal list (13 bits; LL / 16 covers the whole units of the
            // destination whatever its alignment)
            units = LL >> 4;
            packed = bytes | (units << 17);
            sc = packed;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t t = __shfl_up_sync(FULL, sc, d);
                if (lane >= (uint32_t)d) sc += t;
            }
            lits = __ballot_sync(FULL, units != 0u);
        }
        if (lane == 31) {
            c.ex[EX_SCAN + warp] = sc;
            c.ex[EX_LIT + warp] = (uint32_t)__popc(lits);
        }
        carry = n ? c.desc[n - 1u].y : carry;
        __syncthreads();
        sc -= packed;
        uint32_t total = 0, entry = (uint32_t)__popc(lits & ((1u << lane) - 1u)), entries = 0;
#pragma unroll 1
        for (uint32_t j = 0; j < W; j++) {
            const uint32_t t = c.ex[EX_SCAN + j], e = c.ex[EX_LIT + j];
            total += t;
            entries += e;
            if (j < warp) {
                sc += t;
                entry += e;
            }
        }
        const uint32_t base = o + (sc & 0x1ffffu), t0 = sc >> 17;
        o += total & 0x1ffffu;
        if (fin) size_known(o);
        if (busy) {
            const uint32_t d = base + 1u + nll, end = d + LL;
            if (mine || last) {
                dst[base] = (uint8_t)(((LL < 15u ? LL : 15u) << 4) | (ML < 15u ? ML : 15u));
                if (nll) dst[d - 1u] = (uint8_t)((LL - 15u) % 255u);
                if (mine) {
                    dst[end] = (uint8_t)(off & 255u);
                    dst[end + 1u] = (uint8_t)(off >> 8);
                    if (nml) dst[end + 1u + nml] = (uint8_t)((ML - 15u) % 255u);
                }
                // The run's whole 16-byte units [u0, u1) of the slot go to the list;
                // here what is left before them (up to three bytes, then words)
                // and after them (words, then bytes).  A run inside one unit
                // has u0 = u1 at its last word boundary (before the slot's
                // first unit, u1 is -4).
                const uint32_t w0 = (d + 3u) & ~3u, w1 = end & ~3u, by = anchor - d;
                uint32_t u0 = ((d + 4u + 15u) & ~15u) - 4u, u1 = ((end + 4u) & ~15u) - 4u;
                if (u1 < u0 || (int32_t)u1 < 0) u0 = u1 = w0 < end ? w1 : end;
                uint32_t *d32 = reinterpret_cast<uint32_t *>(dst);
#pragma unroll
                for (uint32_t k = 0; k < 3; k++) {
                    if (d + k < w0 && d + k < end) dst[d + k] = src[anchor + k];
                    if (w0 + 4u * k + 4u <= u0) d32[(w0 >> 2) + k] = ld32u(src, by + w0 + 4u * k);
                    if (u1 + 4u * k + 4u <= end) d32[(u1 >> 2) + k] = ld32u(src, by + u1 + 4u * k);
                    const uint32_t b = (w1 > u1 ? w1 : u1) + k;
                    if (b < end) dst[b] = src[by + b];
                }
                if (units)
                    c.desc[entry] = make_uint2(t0 | (((u1 - u0) >> 4) << 16),
                                               (by + u0) | (((u0 + 4u) >> 4) << 16));
            }
            // length bytes of 255, a run of them at a time
#pragma unroll
            for (uint32_t h = 0; h < 2; h++) {
                const uint32_t cnt255 = h ? nml : nll, at = h ? end + 2u : base + 1u;
                for (uint32_t m = __ballot_sync(FULL, cnt255 > 1u); m; m &= m - 1u) {
                    const int l = __ffs(m) - 1;
                    const uint32_t k1 = __shfl_sync(FULL, cnt255, l) - 1u, p = __shfl_sync(FULL, at, l);
#pragma unroll 1
                    for (uint32_t k = lane; k < k1; k += 32) dst[p + k] = 255u;
                }
            }
        }
        __syncthreads();
        // the literal list: each lane finds the entry of its unit by bisection
        const uint32_t nu = total >> 17;
        uint4 *d128 = reinterpret_cast<uint4 *>(dst - 4);
#pragma unroll 1
        for (uint32_t t = tid; t < nu; t += NT) {
            uint32_t e = 0;   // the last entry that starts at or before unit t
#pragma unroll 1
            for (uint32_t h = 0x80000000u >> __clz(entries | 1u); h; h >>= 1)
                if (e + h < entries && (c.desc[e + h].x & 0xffffu) <= t) e += h;
            const uint2 L = c.desc[e];
            const uint32_t k = t - (L.x & 0xffffu);
            if (k < (L.x >> 16)) {
                const uint32_t q = (L.y & 0xffffu) + 16u * k, sh = (q & 3u) * 8u;
                const uint32_t *w = s32 + (q >> 2);
                const uint32_t a = w[0], b = w[1], x = w[2], y = w[3], z = w[4];
                d128[(L.y >> 16) + k] = make_uint4(funnel_r(a, b, sh), funnel_r(b, x, sh),
                                                   funnel_r(x, y, sh), funnel_r(y, z, sh));
            }
        }
        if (fin) break;
        __syncthreads();
    }
    return o;
}

#endif  // __CUDACC__ || BSG_WARP_EMU

}  // namespace bsg
