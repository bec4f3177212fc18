// Compressor (compress_cta.cuh), level 1: cubes.
#include <cuda_runtime.h>

#include "compress_cta.cuh"

namespace bsg {

cudaError_t launch_compress_cta_l1_vis(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    if (a.es == 8) return launch_cta_stream<1, 8, CTA_SAMPLE>(a, max_ctas, s);
    if (a.vis.T % 16u != 0) return launch_cta_stream<1, 4, CTA_SAMPLE>(a, max_ctas, s);
    return launch_cta_stream<1, 4, CTA_GROUP_X>(a, max_ctas, s);
}

}  // namespace bsg
