// Decoder kernels of U8 launches (one translation unit per dtype
// family, so that the kernels compile in parallel).
#include "decode_kernels.cuh"

namespace zipnn {

const void* decode_kernel_u8(int kind, int threads, bool three) { return kernel_handle<ZIPNN_U8>(kind, threads, three); }

}  // namespace zipnn
