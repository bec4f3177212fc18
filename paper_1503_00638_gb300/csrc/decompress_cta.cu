// Decompressor (decompress_cta.cuh): instantiations and dispatch.
#include <cuda_runtime.h>

#include "decompress_cta.cuh"

namespace bsg {

cudaError_t launch_decompress_cta(const CodecArgs &a, cudaStream_t s)
{
    switch (a.es) {
    case 1: return launch_decompress_cta_es<1>(a, s);
    case 2: return launch_decompress_cta_es<2>(a, s);
    case 4: return launch_decompress_cta_es<4>(a, s);
    default: return launch_decompress_cta_es<8>(a, s);
    }
}

}  // namespace bsg
