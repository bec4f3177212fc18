// Compressor (compress_cta.cuh): sizing, dispatch and the level-0 kernels of
// 4-byte elements.
#include <cuda_runtime.h>

#include "compress_cta.cuh"

namespace bsg {

uint32_t compress_cta_max(uint32_t S, uint32_t sms)
{
    // (the larger of the two levels, with the usual tables)
    const uint32_t s0 = cta_plan<0>(S).smem, s1 = cta_plan<1>(S).smem, W = cta_plan<0>(S).W;
    uint32_t p0 = (228u * 1024u) / (s0 + 1024u), p1 = (228u * 1024u) / (s1 + 1024u);
    if (p0 > 32u / W) p0 = 32u / W;
    if (p1 > 32u) p1 = 32u;
    return sms * (p0 > p1 ? p0 : p1 ? p1 : 1u);
}

size_t compress_cta_slots_bytes(uint32_t S, uint32_t ctas)
{
    return (size_t)ctas * 2u * cta_plan<0>(S).slot;
}

bool compress_cta_ok(uint32_t es, uint32_t B) { return cta_shape_ok(es, B); }

cudaError_t launch_compress_cta(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    if (a.level >= 1)
        return a.vis.enabled ? launch_compress_cta_l1_vis(a, max_ctas, s) : launch_compress_cta_l1(a, max_ctas, s);
    if (a.vis.enabled) return launch_compress_cta_vis(a, max_ctas, s);
    switch (a.es) {
    case 1: return launch_compress_cta1(a, max_ctas, s);
    case 2: return launch_compress_cta2(a, max_ctas, s);
    case 4: return launch_cta_stream<0, 4, CTA_PLAIN, 2048, 1024, 512, 4096, 8192>(a, max_ctas, s);
    default: return launch_compress_cta8(a, max_ctas, s);
    }
}

}  // namespace bsg
