// Level-0 compressor (compress_cta.cuh): sizing, dispatch and the kernels of
// 4-byte elements.
#include <cuda_runtime.h>

#include "compress_cta.cuh"

namespace bsg {

uint32_t compress_cta_max(uint32_t S, uint32_t sms)
{
    const CtaPlan plan = cta_plan(S);
    uint32_t per = (228u * 1024u) / (plan.smem + 1024u);
    if (per > 32u / plan.W) per = 32u / plan.W;
    return sms * (per ? per : 1u);
}

size_t compress_cta_slots_bytes(uint32_t S, uint32_t ctas)
{
    return (size_t)ctas * 2u * cta_plan(S).slot;
}

bool compress_cta_ok(uint32_t es, uint32_t B) { return cta_shape_ok(es, B); }

cudaError_t launch_compress_cta(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    if (a.vis.enabled) return launch_compress_cta_vis(a, max_ctas, s);
    switch (a.es) {
    case 1: return launch_compress_cta1(a, max_ctas, s);
    case 2: return launch_compress_cta2(a, max_ctas, s);
    case 4: return launch_cta_stream<4, CTA_PLAIN, 2048, 1024>(a, max_ctas, s);
    default: return launch_compress_cta8(a, max_ctas, s);
    }
}

}  // namespace bsg
