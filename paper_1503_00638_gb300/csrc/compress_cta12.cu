// Level-0 compressor (compress_cta.cuh): 1- and 2-byte elements.
#include <cuda_runtime.h>

#include "compress_cta.cuh"

namespace bsg {

cudaError_t launch_compress_cta1(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    return launch_cta_stream<0, 1, CTA_PLAIN, 8192, 4096, 2048>(a, max_ctas, s);
}

cudaError_t launch_compress_cta2(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    return launch_cta_stream<0, 2, CTA_PLAIN, 4096, 2048, 1024>(a, max_ctas, s);
}

}  // namespace bsg
