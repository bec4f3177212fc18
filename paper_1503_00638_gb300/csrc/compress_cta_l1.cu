// Compressor (compress_cta.cuh), level 1: elements.
#include <cuda_runtime.h>

#include "compress_cta.cuh"

namespace bsg {

cudaError_t launch_compress_cta_l1(const CodecArgs &a, uint32_t max_ctas, cudaStream_t s)
{
    switch (a.es) {
    case 1: return launch_cta_stream<1, 1, CTA_PLAIN>(a, max_ctas, s);
    case 2: return launch_cta_stream<1, 2, CTA_PLAIN>(a, max_ctas, s);
    case 4: return launch_cta_stream<1, 4, CTA_PLAIN>(a, max_ctas, s);
    default: return launch_cta_stream<1, 8, CTA_PLAIN>(a, max_ctas, s);
    }
}

}  // namespace bsg
