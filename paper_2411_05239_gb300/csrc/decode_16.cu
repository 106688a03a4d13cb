// Decoder kernels of 16-bit (BF16 and FP16) launches (one translation unit per dtype
// family, so that the kernels compile in parallel).
#include "decode_kernels.cuh"

namespace zipnn {

const void* decode_kernel_16(int kind, int threads, bool three) { return kernel_handle<ZIPNN_BF16>(kind, threads, three); }

}  // namespace zipnn
