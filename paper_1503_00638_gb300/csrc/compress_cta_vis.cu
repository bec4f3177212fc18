// Level-0 compressor (compress_cta.cuh): cubes as 4-byte components.
#include <cuda_runtime.h>

#include "compress_cta.cuh"

namespace bsg {

cudaError_t launch_compress_cta_vis(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    if (a.es == 8) return launch_compress_cta_vis8(a, max_ctas, s);
    // groups of 16 samples must not straddle products
    if (a.vis.T % 16u != 0) return launch_compress_cta_sample(a, max_ctas, s);
    if (a.vis.is_int || a.vis.cft || a.vis.qtab) return launch_compress_cta_group_x(a, max_ctas, s);
    return launch_cta_stream<0, 4, CTA_GROUP, 2048, 1024>(a, max_ctas, s);
}

}  // namespace bsg
