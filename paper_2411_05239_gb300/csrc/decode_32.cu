// Decoder kernels of FP32 launches (one translation unit per dtype
// family, so that the kernels compile in parallel).
#include "decode_kernels.cuh"

namespace zipnn {

const void* decode_kernel_32(int kind, int threads, bool three) { return kernel_handle<ZIPNN_FP32>(kind, threads, three); }

}  // namespace zipnn
