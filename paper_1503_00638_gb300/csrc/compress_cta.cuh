// The compress kernel: [gather ->] round -> bit-transpose -> LZ4 ->
// placement of one block per CTA step (Sec. 4.2.1, Sec. 6 steps 1-5), for
// every element size, every block size up to 64 KiB whose bit-rows are whole
// words (cta_shape_ok), and the shortened last block of such a stream.
#pragma once

#include "codec.cuh"
#include "lz4_cta.cuh"
#include "shuffle_cta.cuh"

namespace bsg {

// How a block's elements are prepared before the transpose.
enum CtaMode {
    CTA_PLAIN,    // as they are
    CTA_GROUP,    // float32 cube, constant c, time axis a multiple of 16: in
                  // registers, a thread's 32 words being 16 samples of one product
    CTA_GROUP_X,  // the same for int32, the compensated c or the full-covariance q
    CTA_SAMPLE    // any time axis and 8-byte samples: in shared memory first
};

// Resident warps per SM of the kernels with a fixed block size of one or two
// warps: 28, with 72 registers a thread.  Larger blocks have 32 at 64 (a CTA more
// per SM counts for more there), as the kernel of any size.
constexpr uint32_t CTA_WARPS_PER_SM = 28;

// Bytes of full blocks of S bytes from which a stream with a shortened last
// block takes two launches: what the fixed block size saves grows with the
// stream, the second launch takes 5 to 8 us.  Walks, all in one launch and in
// two: 64 MiB of 4-byte elements in 2, 4 and 8 KiB blocks 122, 77 and 73 us, and
// 118, 80 and 74 (32 MiB 71, 47 and 46, and 74, 55 and 52; 128 MiB 224, 134 and
// 128, and 205, 127 and 119); 64 MiB in 16 and 32 KiB 68 and 72, and 74 and 79,
// 128 MiB 121 and 126, and 118 and 124.
constexpr uint64_t cta_split_bytes(uint32_t S) { return (S <= 8192u ? 64ull : 128ull) << 20; }

struct CtaPlan {
    uint32_t W;          // warps
    uint32_t tmp;        // bytes of the block buffer
    uint32_t smem;       // dynamic shared memory
    uint32_t slot;       // bytes of a staging slot
};
// Warps of level 1: two units of 128 bytes to a thread.  Its search is one
// warp's work and shared memory, with the hash table in it, holds 16 blocks of
// 8 KiB per SM whatever the warps, so a second warp per block only took
// registers, and what counts is that the search keeps its values in them: 67
// MB of 16-bit walks in 8 KiB blocks take 245 us at 128 registers a thread,
// 305 at 112, 317 at 96, 326 at 80 (the one-warp kernel that wrote each
// sequence before it searched on: 299), 364 us with two warps at 64.
template <int LEVEL>
__host__ __device__ constexpr uint32_t cta_warps_of(uint32_t S)
{
    return LEVEL >= 1 ? (S + 8191u) / 8192u : cta_warps(S);
}

// Nodes for the parse graph of a kernel with a fixed block size of S bytes (0:
// the usual number, 64 a warp).  Cubes have few, other data up to one to 28
// bytes.  64 MiB of which one byte in 33 is not zero has 72 nodes to 2 KiB and
// 290 to 8 KiB on average: 450 us in blocks of 2 KiB and 400 in 8 KiB with 64 a
// warp (the one-warp encoder with its 128: 282 and 381), 190 and 260 so.  At 4
// KiB, where 64 are no slower than that encoder was (242 and 371 us), more
// would cost other data shared memory and L1 (walks 79 -> 81 us; int32 cube in
// the instrument's order 252 -> 260).
template <int MODE>
__host__ __device__ constexpr uint32_t cta_fixed_cap(uint32_t S)
{
    if (MODE != CTA_PLAIN) return 0;
    return S <= 2048u ? 96u : S > 4096u && S <= 8192u ? 320u : 0u;
}

// (cap: nodes of level 0's tables, 0 for the usual number)
template <int LEVEL>
__host__ __device__ constexpr CtaPlan cta_plan(uint32_t S, uint32_t cap = 0)
{
    const uint32_t W = cta_warps_of<LEVEL>(S), tmp = r16(S + 16u);
    return CtaPlan{W, tmp, tmp + r16(cta_scratch_bytes<LEVEL>(W, cta_hbits(S), cap)) + 16u,
                   r16(4u + lz4b(S) + 32u)};
}

// Round 16 complex samples in registers (v[m] = component (m + 4 rot) mod 32
// of the group) with the constant c.  Per component two additions, the sign
// and one OR: whether |x| was below 2^(k+23) (and a number) is not tested
// component by component but once per group, from the exponents of the
// sums |x| + 2^(k+23), which then all equal that of 2^(k+23).  Returns false
// when some component needs the full rule (values beyond 2^(k+23), NaN,
// infinities, an unusable q): the registers are then garbage and the caller
// rounds the group sample by sample.
BSG_D bool cta_round_group(const VisParams &P, uint32_t (&v)[32], uint32_t rot, const float *ai,
                           const float *aj, bool is_auto)
{
    const float cc = is_auto ? P.c2 : P.c;
    uint32_t big = 0, worst = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const uint32_t c = (k + rot) & 7u;  // samples 2 c and 2 c + 1
        const float2 Ai = __ldg(reinterpret_cast<const float2 *>(ai + 2 * c));
        const float2 Aj = __ldg(reinterpret_cast<const float2 *>(aj + 2 * c));
#pragma unroll
        for (int s = 0; s < 2; s++) {
            const uint32_t Q = __float_as_uint(
                __fmul_rn(__fmul_rn(cc, s ? Ai.y : Ai.x), s ? Aj.y : Aj.x));
            // magic_bits(Q), the constant 86 << 23 folded in before the shift
            const uint32_t Tb = ((Q + 0x007fffffu + (86u << 24)) >> 1) & 0x7f800000u;
            const float T = __uint_as_float(Tb);
            const uint32_t u = Q - 0x00800000u;   // q_usable: below 0x7f000000
            worst = worst > u ? worst : u;
#pragma unroll
            for (int h = 0; h < 2; h++) {
                if (h && is_auto) continue;   // the imaginary part of an auto stays
                uint32_t &w = v[4 * k + 2 * s + h];
                const float t = __fadd_rn(fabsf(__uint_as_float(w)), T);
                big |= __float_as_uint(t) ^ Tb;
                w = __float_as_uint(__fsub_rn(t, T)) | (w & 0x80000000u);
            }
        }
    }
    return (big & 0x7f800000u) == 0u && worst < 0x7f000000u;
}

template <int ES, int MODE>
struct CtaRound {
    const VisParams *P;
    uint8_t *buf;
    uint32_t c_blk;   // complex index of the block's first sample
    BSG_D void operator()(uint32_t g, uint32_t (&v)[32]) const
    {
        if (MODE == CTA_GROUP_X) {
            const VisGroupRound round{P, c_blk};
            round(g, v);
        } else if (MODE == CTA_GROUP) {
            const uint32_t cg = c_blk + 16u * g;
            const uint32_t fp = fastdiv(cg, P->dT), t0 = cg - fp * P->T;
            const uint32_t f = fastdiv(fp, P->dP), p = fp - f * P->P;
            const uint32_t ij = __ldg(P->pairs + p), i = ij & 0xffffu, j = ij >> 16;
            const float *ai = P->autos + (size_t)(f * P->n_in + i) * P->T + t0;
            const float *aj = P->autos + (size_t)(f * P->n_in + j) * P->T + t0;
            if (!cta_round_group(*P, v, g & 7u, ai, aj, i == j)) {
                // rare: the group's samples again from shared memory, by the full rule
                uint4 *grp = reinterpret_cast<uint4 *>(buf + 128u * g);
                const float cc = i == j ? P->c2 : P->c;
#pragma unroll 1
                for (uint32_t c = 0; c < 16; c++) {
                    const float q = __fmul_rn(__fmul_rn(cc, __ldg(ai + c)), __ldg(aj + c));
                    float *x = reinterpret_cast<float *>(grp) + 2u * c;
                    x[0] = reduce_one(x[0], q);
                    if (i != j) x[1] = reduce_one(x[1], q);
                }
#pragma unroll
                for (uint32_t k = 0; k < 8; k++) {
                    const uint4 q = grp[(k + g) & 7u];
                    v[4 * k] = q.x;
                    v[4 * k + 1] = q.y;
                    v[4 * k + 2] = q.z;
                    v[4 * k + 3] = q.w;
                }
            }
        }
    }
};

// Start loading block `tile` (bytes long) into buf; true when a bulk copy is
// in flight on `bar`.  The ragged end (< 16 bytes, a shortened last block)
// comes by plain loads.
BSG_D bool cta_load(uint8_t *buf, const uint8_t *src, uint32_t bytes, uint64_t *bar)
{
    const uint32_t bulk = bytes & ~15u;
    if (threadIdx.x == 0 && bulk) {
        mbar_arrive_expect_tx(bar, bulk);
        bulk_g2s(buf, src, bulk, bar);
    }
    if (threadIdx.x < (bytes & 15u)) buf[bulk + threadIdx.x] = src[bulk + threadIdx.x];
    return bulk != 0u;
}

// Samples c0 .. c0 + n - 1 of a time-slowest cube into time-fastest order.  A
// block holds n / T series, whose samples of one time are neighbours in the
// input: consecutive threads take consecutive series, so a request reads
// whole sectors.  Time axes longer than half a block go sample by sample.
// With a time axis of whole 16-sample groups the group form below is used.
BSG_D void cta_gather_samples(const CodecArgs &a, uint8_t *buf, uint32_t c0, uint32_t n)
{
    const VisParams &P = a.vis;
    const uint2 *src = reinterpret_cast<const uint2 *>(a.in);
    uint2 *d = reinterpret_cast<uint2 *>(buf);
    const uint32_t tid = threadIdx.x, NT = blockDim.x;
    if (cta_gather_single(P.T, n)) {
#pragma unroll 1
        for (uint32_t k = tid; k < n; k += NT) {
            const uint32_t c = c0 + k, s = fastdiv(c, P.dT), t = c - s * P.T;
            d[k] = __ldg(src + (uint64_t)t * P.FP + s);
        }
        return;
    }
    const uint32_t s0 = fastdiv(c0, P.dT), ns = fastdiv(c0 + n - 1u, P.dT) - s0 + 1u;
    const uint32_t dt = NT / ns, ds = NT - dt * ns;
    uint32_t t = tid / ns, s = tid - t * ns;
    const uint32_t lead = c0 - s0 * P.T;   // samples of the first series before the block
#pragma unroll 2
    for (uint32_t it = tid; it < P.T * ns; it += NT) {
        const uint32_t k = s * P.T + t - lead;   // wraps below zero for t < lead in series 0
        if (k < n) d[k] = __ldg(src + (uint64_t)t * P.FP + s0 + s);
        t += dt;
        s += ds;
        if (s >= ns) {
            s -= ns;
            t++;
        }
    }
}

// A time axis that is a multiple of 16: thread q takes 16-sample series
// groups q, q + NT, ... (neighbouring threads, neighbouring series), their
// 16-byte chunks in an order rotated by lane / 4: at every step the four lanes
// of one 32-byte sector of neighbouring series read the same time row, and the
// chunks the 32 lanes store fall in eight different bank groups.
BSG_D void cta_gather_groups(const CodecArgs &a, uint8_t *buf, uint32_t c0, uint32_t n)
{
    const VisParams &P = a.vis;
    const uint64_t row = P.FP;
    const uint2 *src = reinterpret_cast<const uint2 *>(a.in);
    const uint32_t m = (threadIdx.x >> 2) & 7u;
#pragma unroll 1
    for (uint32_t q = threadIdx.x; q < n / 16u; q += blockDim.x) {
        const uint32_t c = c0 + 16u * q, s = fastdiv(c, P.dT), t0 = c - s * P.T;
        const uint2 *p = src + (uint64_t)t0 * row + s;
        uint4 *d = reinterpret_cast<uint4 *>(buf + (size_t)128 * q);
#pragma unroll
        for (uint32_t k = 0; k < 8; k++) {
            const uint32_t x = (k + m) & 7u;
            const uint2 u = __ldg(p + (uint64_t)(2 * x) * row);
            const uint2 v = __ldg(p + (uint64_t)(2 * x + 1) * row);
            d[x] = make_uint4(u.x, u.y, v.x, v.y);
        }
    }
}

// Round n samples from complex index c0 in shared memory, two at a time when
// the time axis is even (c0 and n then are).
BSG_D void cta_round_samples(uint8_t *buf, uint32_t c0, uint32_t n, const VisParams &P)
{
    const uint32_t tid = threadIdx.x, NT = blockDim.x;
    if ((P.T & 1u) == 0) {
        uint4 *b4 = reinterpret_cast<uint4 *>(buf);
#pragma unroll 1
        for (uint32_t k = tid; k < n / 2u; k += NT) {
            const uint32_t c = c0 + 2u * k;
            const uint32_t fp = fastdiv(c, P.dT), t = c - fp * P.T;
            const uint32_t f = fastdiv(fp, P.dP), p = fp - f * P.P;
            b4[k] = reduce_pair(b4[k], __ldg(P.pairs + p), f, t, P);
        }
    } else {
        uint2 *b2 = reinterpret_cast<uint2 *>(buf);
#pragma unroll 1
        for (uint32_t k = tid; k < n; k += NT) {
            const uint32_t c = c0 + k;
            const uint32_t fp = fastdiv(c, P.dT), t = c - fp * P.T;
            const uint32_t f = fastdiv(fp, P.dP), p = fp - f * P.P;
            b2[k] = reduce_sample(b2[k], __ldg(P.pairs + p), f, t, P);
        }
    }
}

// Copy len bytes from 16-byte aligned global `s` (a staging slot, in L2) to
// global `g` (any alignment), as copy_out does from shared memory.  (Two to
// four chunks per thread in flight: no faster, the registers cost as much.)
BSG_D void cta_copy_out(const uint8_t *s, uint8_t *g, uint32_t len)
{
    const uint32_t tid = fresh_tid(), NT = blockDim.x;
    uint32_t head = (uint32_t)((16u - ((uintptr_t)g & 15u)) & 15u);
    if (head > len) head = len;
    if (tid < head) g[tid] = __ldcg(s + tid);
    const uint32_t nchunk = (len - head) / 16u;
    const uint4 *s4 = reinterpret_cast<const uint4 *>(s);
    const uint32_t q = (head >> 2) & 3u, sh = (head & 3u) * 8u;
#pragma unroll 1
    for (uint32_t c = tid; c < nchunk; c += NT) {
        const uint32_t so = head + 16u * c;
        const uint4 A = __ldcg(s4 + (so >> 4)), B = __ldcg(s4 + (so >> 4) + 1);
        // the five words from word q of A on, moved down by whole words first
        uint32_t w0 = A.x, w1 = A.y, w2 = A.z, w3 = A.w, w4 = B.x;
        if (q & 1u) {
            w0 = w1; w1 = w2; w2 = w3; w3 = w4; w4 = B.y;
        }
        if (q & 2u) {
            w0 = w2; w1 = w3; w2 = w4; w3 = (q & 1u) ? B.z : B.y; w4 = (q & 1u) ? B.w : B.z;
        }
        *reinterpret_cast<uint4 *>(g + so) =
            make_uint4(funnel_r(w0, w1, sh), funnel_r(w1, w2, sh), funnel_r(w2, w3, sh),
                       funnel_r(w3, w4, sh));
    }
    const uint32_t k = head + 16u * nchunk + tid;
    if (k < len) g[k] = __ldcg(s + k);
}

// Block `tile` from its staging slot (4 + cs bytes) to stream offset D, with
// its index entry.
BSG_D void cta_place(const CodecArgs &a, uint32_t tile, const uint8_t *slot, uint32_t cs, uint64_t D)
{
    if (D + 4 + cs > a.out_cap) {
        if (threadIdx.x == 0) set_status(a.status, BSGPU_ERR_SPACE);
        return;
    }
    cta_copy_out(slot, a.out + D, 4 + cs);
    if (a.block_offsets && threadIdx.x == 0) a.block_offsets[tile] = D;
}

// Exclusive prefix of a block whose size is published, as lookback_resolve,
// but at most `looks` looks in vain: LB_UNKNOWN then.  With a status word the
// wait is the last one: when it runs out, or another block's has (the stream is
// lost then, and one limit is all that the call may wait), it reports
// BSGPU_ERR_TIMEOUT and publishes what it has added up, so that no successor
// waits for this block.  (Looking at 64, 128 or 256 predecessors per step
// instead of 32 changed nothing: 224-234 us on the 33024 blocks below; sums of
// groups of 128 blocks by atomics, which thousands of warps read, kept the
// atomics waiting: 268 to 970 us.)
constexpr uint64_t LB_UNKNOWN = ~0ull;

BSG_D uint64_t lookback_some(uint64_t *state, uint32_t tile, uint64_t agg, uint32_t looks,
                             int *status, uint32_t lane)
{
    uint64_t excl = 0;
    uint32_t spins = 0;
    bool found = true;
    int64_t base = (int64_t)tile - 1;   // blocks base, base - 1, ... are still to be added
    for (bool done = tile == 0; !done;) {
        const int64_t idx = base - (int64_t)lane;
        uint64_t v = idx >= 0 ? ld_relaxed_u64(state + idx) : LB_FP;
#ifdef BSG_TEST_LOOKBACK_STALL
        if (idx >= 0) v = 0;   // test builds only, as in lookback_resolve
#endif
        const uint32_t flag = (uint32_t)(v >> 62);
        const uint32_t pm = __ballot_sync(FULL, flag == 2), im = __ballot_sync(FULL, flag == 0);
        const uint32_t first = pm ? (uint32_t)(__ffs(pm) - 1) : 32u;
        if (im & (first >= 32u ? FULL : (1u << first) - 1u)) {
            if (++spins >= looks ||
                (status && spins % 256u == 0 && __any_sync(FULL, *(volatile int *)status != 0))) {
                if (!status) return LB_UNKNOWN;
                found = false;
                break;
            }
            if (spins > 4096) __nanosleep(100);
            continue;
        }
        // the sizes of 32 blocks add up to less than 2^32
        excl += __reduce_add_sync(FULL, lane < first ? (uint32_t)v : 0u);
        if (pm) {
            excl += __shfl_sync(FULL, v, first) & LB_VM;
            done = true;
        }
        base -= 32;
    }
    if (tile && lane == 0) st_relaxed_u64(state + tile, LB_FP | (excl + agg));
    if (!found) {
        if (lane == 0) set_status(status, BSGPU_ERR_TIMEOUT);
        return LB_UNKNOWN;
    }
    return excl;
}

// One block at a time per CTA (persistent, tiles in order from a counter):
// the block is transposed in place through registers and encoded into a
// staging slot in global memory (it stays in L2); its size is published as
// soon as the parse knows it, and the PREVIOUS block is placed while the next
// one loads: by then its predecessors have long published theirs, so the
// look-back rarely waits.
//
// What bounds it: the latency of its stages and instruction issue, about
// evenly (CHIME-shaped cube, 256 frequencies, 33024 blocks of 8 KiB: 217 us,
// issue active 57 %, ALU 54 %, shared-memory pipe 49 %, DRAM 25 %; 24, 28 or
// 32 warps per SM make no difference).  The one-warp kernel it replaces took
// 290 us there.  Whole cube, 1.08 GB: 1.10 -> 0.86 ms; 268 MB of float64 in
// 32 KiB blocks, which took a kernel of two buffers per warp: 0.88 -> 0.18 ms.
//
// BC: the block size in elements when it is one of the usual ones (4 and 8
// KiB; but for cubes 2 KiB and, of 4- and 8-byte elements, 16 and 32; full blocks
// only), else 0 for any size and for a shortened last block.  With the size known the strides of
// the bit-rows, the loops over the warps and the tables' places are constants
// (int32 cube, time slowest, as 8-byte samples in 4 KiB blocks, 127 MB: 279 ->
// 253 us; 268 MB of float64 in 32 KiB blocks: 206 -> 182 us).  TS: a
// time-slowest cube.
template <int LEVEL, int ES, int MODE, uint32_t BC, bool TS>
BSG_D void compress_cta_body(const CodecArgs &a)
{
    extern __shared__ __align__(128) uint8_t sm[];
    const uint32_t W = BC ? cta_warps(BC * ES) : blockDim.x >> 5;
    constexpr uint32_t CAP = BC ? cta_fixed_cap<MODE>(BC * ES) : 0u;
    const CtaPlan plan = cta_plan<LEVEL>((BC ? BC : a.B) * ES, CAP);
    const uint32_t hbits = cta_hbits((BC ? BC : a.B) * ES);
    uint8_t *buf = sm;
    const CtaScratch c = cta_scratch<LEVEL>(sm + plan.tmp, W, hbits, CAP);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + plan.smem - 16u);
    uint32_t *next = c.ex + EX_CTL + 2;            // the next tile
    uint64_t *excl = reinterpret_cast<uint64_t *>(c.ex + EX_CTL + 4);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
        *next = a.tile_begin + atomicAdd(a.tile_counter, 1u);
    }
    __syncthreads();
    uint32_t tile = *next, parity = 0;
    uint8_t *slot0 = a.slots + (size_t)(2 * blockIdx.x) * plan.slot, *slot1 = slot0 + plan.slot;
    uint32_t ptile = ~0u, pcs = 0;                 // the block waiting to be placed, in slot1
    bool pend = false;
    auto elems = [&](uint32_t t) { return BC ? BC : block_elems_of(a, t); };
    if (!TS && tile < a.tile_end)
        pend = cta_load(buf, a.in + (uint64_t)tile * a.B * ES, elems(tile) * ES, bar);
    for (;;) {
        const bool work = tile < a.tile_end;
        const uint32_t tid = fresh_tid(), lane = tid & 31u, warp = tid >> 5;
        uint32_t cs = 0, nxt = tile;
        if (work) {
            const uint32_t Bb = elems(tile), S = Bb * ES;
            const uint32_t c0 = (uint32_t)(((uint64_t)tile * a.B * ES) >> 3);   // first complex sample
            if (pend) {
                if (!mbar_wait_bounded(bar, parity) && tid == 0) set_status(a.status, BSGPU_ERR_TIMEOUT);
                parity ^= 1u;
            }
            if (TS) {
                if (a.vis.T % 16u == 0 && S % 128u == 0)
                    cta_gather_groups(a, buf, c0, S / 8u);
                else
                    cta_gather_samples(a, buf, c0, S / 8u);
            }
            if (TS || (S & 15u)) __syncthreads();   // what plain stores brought
            if (MODE == CTA_SAMPLE) {
                cta_round_samples(buf, c0, S / 8u, a.vis);
                __syncthreads();
            }
            constexpr uint32_t UPT = LEVEL >= 1 ? 2 : 1;   // units per thread
            uint32_t v[UPT][32];
            const uint32_t units = cta_units<ES>(Bb);
#pragma unroll
            for (uint32_t k = 0; k < UPT; k++)
                if (tid + 32u * W * k < units)
                    cta_get_rows<ES>(buf, Bb, tid + 32u * W * k, v[k], CtaRound<ES, MODE>{&a.vis, buf, c0});
            __syncthreads();
#pragma unroll
            for (uint32_t k = 0; k < UPT; k++)
                if (tid + 32u * W * k < units) cta_put_rows<ES>(buf, Bb, tid + 32u * W * k, v[k]);
            __syncthreads();
            if (!cta_rows_whole<ES>(Bb)) cta_pack_rows<ES>(buf, Bb);
            const uint32_t *s32 = reinterpret_cast<const uint32_t *>(buf);
            const uint32_t rowlen = Bb / 8u, R = (rowlen & 3u) ? 0u : rowlen / 4u;
            if (LEVEL >= 1) {
                // (no bitmaps)
            } else if ((ES == 4 || ES == 8) && Bb % 1024u == 0) {
                // a warp's rows are whole bitmap words and still in its registers:
                // compare each with the row above and the word to the left
                const uint32_t h = ES == 8 && tid >= R ? 1u : 0u, g = tid - h * R;
                if (tid < units) {
                    uint32_t w = 32u * h * R + g;
                    uint32_t up = h ? s32[w - R] : ~v[0][0];
                    uint2 *E = c.E + (w >> 5);
#pragma unroll
                    for (int r = 0; r < 32; r++) {
                        const uint32_t left = r || w ? s32[(int)w - 1] : ~v[0][0];
                        const uint32_t row = __ballot_sync(FULL, v[0][r] == up);
                        const uint32_t run = __ballot_sync(FULL, v[0][r] == left);
                        if (lane == 0) *E = make_uint2(row, run);
                        up = v[0][r];
                        w += R;
                        E += R >> 5;
                    }
                }
            } else {
                cta_eq_bitmaps<BC && ES <= 2 ? 8 : 1>(s32, S / 4u, R, c, W);
            }
            if (LEVEL == 0) __syncthreads();
            cs = cta_lz4_encode<LEVEL>(
                buf, S, rowlen, slot0 + 4, c, W, hbits,
                [&](uint32_t size) {
                    if (tid == 0) {
                        lookback_publish(a.tile_state, tile, 4ull + size, 0);
                        put_be32(slot0, size);
                        *next = a.tile_begin + atomicAdd(a.tile_counter, 1u);
                    }
                },
                [&] {   // the previous block's place, while this warp has nothing else to do
                    if (ptile != ~0u) {
                        const uint64_t x = lookback_some(a.tile_state, ptile, 4ull + pcs, 8u, nullptr, lane);
                        if (lane == 0) *excl = x;
                    }
                });
            fence_proxy_async_smem();   // the reads of buf before the next bulk write
            __syncthreads();
            nxt = *next;
            pend = false;
            if (!TS && nxt < a.tile_end)
                pend = cta_load(buf, a.in + (uint64_t)nxt * a.B * ES, elems(nxt) * ES, bar);
        }
        if (ptile != ~0u) {
            if (W == 1 || !work || *excl == LB_UNKNOWN) {
                __syncthreads();   // everyone has seen *excl
                if (warp == 0) {
                    const uint64_t x = lookback_some(a.tile_state, ptile, 4ull + pcs, 1u << 21, a.status, lane);
                    if (lane == 0) *excl = x;
                }
                __syncthreads();
            }
            if (*excl != LB_UNKNOWN) cta_place(a, ptile, slot1, pcs, 12 + *excl);
        }
        if (!work) break;
        ptile = tile;
        pcs = cs;
        uint8_t *t = slot0;
        slot0 = slot1;
        slot1 = t;
        tile = nxt;
    }
    // (outside the loop, where it costs the other blocks no registers)
    if (a.tile_begin == 0 && blockIdx.x == 0 && threadIdx.x < 32)
        write_chunk_header(a.out, a.n_elem * ES, a.B * ES, threadIdx.x);
    if (ptile + 1u == a.nb && threadIdx.x < 32) {
        if (*excl != LB_UNKNOWN)
            compress_place_end(a, 12 + *excl + 4 + pcs, threadIdx.x);
        else if (threadIdx.x == 0)
            *a.out_bytes = 0;   // (the status tells)
    }
}

template <int ES, int MODE, uint32_t BC, bool TS>
__global__ void __launch_bounds__(BC ? 32 * cta_warps(BC *ES) : 32 * CTA_MAX_WARPS,
                                  BC ? (cta_warps(BC *ES) > 2 ? 32u : CTA_WARPS_PER_SM) / cta_warps(BC *ES) : 2)
    compress_cta_kernel(const __grid_constant__ CodecArgs a)
{
    compress_cta_body<0, ES, MODE, BC, TS>(a);
}

// Level 1: shared memory bounds its CTAs, so a thread may have more registers
// (see cta_warps_of).
constexpr int CTA_L1_REGS = 128;

template <int ES, int MODE, bool TS>
__global__ void __maxnreg__(CTA_L1_REGS)
    compress_cta_l1_kernel(const __grid_constant__ CodecArgs a)
{
    compress_cta_body<1, ES, MODE, 0, TS>(a);
}

// Tiles [a.tile_begin, a.tile_end) with as many CTAs as fit, at most max_ctas.
template <int LEVEL, int ES, int MODE, uint32_t BC, bool TS = false>
cudaError_t launch_cta(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    const CtaPlan plan = cta_plan<LEVEL>(a.B * ES, BC ? cta_fixed_cap<MODE>(BC * ES) : 0u);
    auto kernel = compress_cta_kernel<ES, MODE, BC, TS>;
    if constexpr (LEVEL >= 1) kernel = compress_cta_l1_kernel<ES, MODE, TS>;
    const cudaError_t e = allow_smem(kernel, plan.smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 148, per = 1;
    if (cudaGetDevice(&dev) == cudaSuccess)
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, (int)(32 * plan.W), plan.smem) !=
            cudaSuccess || per < 1)
        per = 1;
    uint64_t grid = (uint64_t)sms * (uint32_t)per;
    if (grid > max_ctas) grid = max_ctas;
    if (grid > a.tile_end - a.tile_begin) grid = a.tile_end - a.tile_begin;
    kernel<<<(uint32_t)grid, 32 * plan.W, plan.smem, s>>>(a);
    return cudaGetLastError();
}

// The whole stream: full blocks of a usual size through their own kernel and
// a shortened last block after them; other sizes, and streams short enough
// that a second launch costs more than constant strides give, through the
// general one.
template <int LEVEL, int ES, int MODE, bool TS, uint32_t... BCS>
cudaError_t launch_cta_order(const CodecArgs &a0, uint32_t max_ctas, cudaStream_t s)
{
    CodecArgs a = a0;
    const uint32_t nfull = a.nb - (a.last_B != a.B ? 1u : 0u);
    a.tile_begin = 0;
    a.tile_end = a.nb;
    if (sizeof...(BCS) != 0 && (nfull == a.nb || (uint64_t)nfull * a.B * ES >= cta_split_bytes(a.B * ES))) {
        cudaError_t e = cudaErrorNotReady;   // no such kernel
        a.tile_end = nfull;
        ((a.B == BCS ? (void)(e = launch_cta<LEVEL, ES, MODE, BCS, TS>(a, max_ctas, s)) : (void)0), ...);
        if (e == cudaSuccess) {
            if (nfull == a.nb) return e;
            a.tile_begin = nfull;
            a.tile_counter = a.tile_counter + 1;
        } else if (e != cudaErrorNotReady) {
            return e;
        }
        a.tile_end = a.nb;
    }
    return launch_cta<LEVEL, ES, MODE, 0, TS>(a, max_ctas, s);
}

template <int LEVEL, int ES, int MODE, uint32_t... BCS>
cudaError_t launch_cta_stream(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    if constexpr (MODE != CTA_PLAIN)
        if (a.vis.tslow) return launch_cta_order<LEVEL, ES, MODE, true, BCS...>(a, max_ctas, s);
    return launch_cta_order<LEVEL, ES, MODE, false, BCS...>(a, max_ctas, s);
}

}  // namespace bsg
