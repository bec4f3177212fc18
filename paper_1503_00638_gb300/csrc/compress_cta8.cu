// Level-0 compressor (compress_cta.cuh): 8-byte elements, cubes as 8-byte samples.
#include <cuda_runtime.h>

#include "compress_cta.cuh"

namespace bsg {

cudaError_t launch_compress_cta8(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    return launch_cta_stream<0, 8, CTA_PLAIN, 1024, 512, 256, 2048, 4096>(a, max_ctas, s);
}

cudaError_t launch_compress_cta_vis8(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    return launch_cta_stream<0, 8, CTA_SAMPLE, 1024, 512>(a, max_ctas, s);
}

}  // namespace bsg
