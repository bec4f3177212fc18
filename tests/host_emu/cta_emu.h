// Host emulation of one CTA for CPU tests: a std::thread per CUDA thread, a
// barrier per warp for the warp collectives and one for __syncthreads.
#pragma once
#include <atomic>
#include <barrier>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <memory>
#include <thread>
#include <vector>
#include <vector_types.h>      // uint4 and friends; defines __host__ / __device__ as no-ops
#include <vector_functions.h>
#define BSG_WARP_EMU 1
struct EmuDim { unsigned x; };
inline thread_local EmuDim threadIdx;
inline EmuDim blockDim;
struct EmuWarp {
    std::barrier<> bar{32};
    uint32_t v[32];
};
struct EmuCta {
    std::vector<std::unique_ptr<EmuWarp>> warps;
    std::unique_ptr<std::barrier<>> bar;
};
inline EmuCta *g_cta;
inline EmuWarp &emu_warp() { return *g_cta->warps[threadIdx.x >> 5]; }
inline void __syncthreads() { g_cta->bar->arrive_and_wait(); }
inline void __syncwarp(unsigned = 0xffffffffu) { emu_warp().bar.arrive_and_wait(); }
template <class F> inline uint32_t emu_exchange(uint32_t mine, F take)
{
    EmuWarp &w = emu_warp();
    w.v[threadIdx.x & 31u] = mine;
    w.bar.arrive_and_wait();
    const uint32_t r = take(w.v, threadIdx.x & 31u);
    w.bar.arrive_and_wait();
    return r;
}
inline uint32_t __ballot_sync(uint32_t, int p)
{
    return emu_exchange(p ? 1u : 0u, [](const uint32_t *v, uint32_t) {
        uint32_t r = 0;
        for (int i = 0; i < 32; i++) r |= v[i] << i;
        return r;
    });
}
inline uint32_t __shfl_sync(uint32_t, uint32_t x, int src)
{
    return emu_exchange(x, [=](const uint32_t *v, uint32_t) { return v[src & 31]; });
}
inline uint32_t __shfl_up_sync(uint32_t, uint32_t x, unsigned d)
{
    return emu_exchange(x, [=](const uint32_t *v, uint32_t l) { return l >= d ? v[l - d] : x; });
}
inline uint32_t __shfl_down_sync(uint32_t, uint32_t x, unsigned d)
{
    return emu_exchange(x, [=](const uint32_t *v, uint32_t l) { return l + d < 32 ? v[l + d] : x; });
}
inline uint32_t __match_any_sync(uint32_t, uint32_t x)
{
    return emu_exchange(x, [=](const uint32_t *v, uint32_t) {
        uint32_t r = 0;
        for (int i = 0; i < 32; i++) r |= (uint32_t)(v[i] == x) << i;
        return r;
    });
}
inline int __ffs(uint32_t x) { return x ? __builtin_ctz(x) + 1 : 0; }
inline int __popc(uint32_t x) { return __builtin_popcount(x); }
inline int __clz(uint32_t x) { return x ? __builtin_clz(x) : 32; }
inline uint32_t atomicOr(uint32_t *p, uint32_t v) { return __atomic_fetch_or(p, v, __ATOMIC_RELAXED); }
inline void emu_check_aligned4(const void *p)
{
    if ((uintptr_t)p & 3u) {
        fprintf(stderr, "misaligned 4-byte access base %p\n", p);
        abort();
    }
}
namespace bsg { inline uint32_t lanemask_lt() { return (1u << (threadIdx.x & 31u)) - 1u; } }
inline void run_cta(unsigned threads, const std::function<void()> &f)
{
    EmuCta ctx;
    ctx.bar = std::make_unique<std::barrier<>>((std::ptrdiff_t)threads);
    for (unsigned w = 0; w < threads / 32; w++) ctx.warps.push_back(std::make_unique<EmuWarp>());
    g_cta = &ctx;
    blockDim.x = threads;
    std::vector<std::thread> t;
    for (unsigned i = 0; i < threads; i++) t.emplace_back([&, i] { threadIdx.x = i; f(); });
    for (auto &x : t) x.join();
}
