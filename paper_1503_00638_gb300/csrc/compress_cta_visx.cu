// Level-0 compressor (compress_cta.cuh): cubes as 4-byte components, int32, the
// compensated c or the full-covariance q, and any time axis.
#include <cuda_runtime.h>

#include "compress_cta.cuh"

namespace bsg {

cudaError_t launch_compress_cta_group_x(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    return launch_cta_stream<0, 4, CTA_GROUP_X, 2048, 1024>(a, max_ctas, s);
}

cudaError_t launch_compress_cta_sample(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    return launch_cta_stream<0, 4, CTA_SAMPLE, 2048, 1024>(a, max_ctas, s);
}

}  // namespace bsg
