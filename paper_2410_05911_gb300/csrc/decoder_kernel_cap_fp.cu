// decoder_kernel_cap_fp.cu -- instantiations of the decoder kernel with the integer-core capture for warp-task
// attention (full-precision bf16 linears, ReLU and GELU); the plain decode runs the instantiations without it.
#include "decoder_kernel.cuh"

namespace aecct {

template cudaError_t launch_decode<128, 1, 0, 1, 1>(const DecodeParams &, cudaStream_t);
template cudaError_t launch_decode<128, 1, 1, 1, 1>(const DecodeParams &, cudaStream_t);
template cudaError_t launch_decode<32, 1, 0, 1, 1>(const DecodeParams &, cudaStream_t);
template cudaError_t launch_decode<32, 1, 1, 1, 1>(const DecodeParams &, cudaStream_t);
template cudaError_t launch_decode<32, 3, 0, 1, 1>(const DecodeParams &, cudaStream_t);
template cudaError_t launch_decode<32, 3, 1, 1, 1>(const DecodeParams &, cudaStream_t);
template cudaError_t launch_decode<64, 1, 0, 1, 1>(const DecodeParams &, cudaStream_t);
template cudaError_t launch_decode<64, 1, 1, 1, 1>(const DecodeParams &, cudaStream_t);
template cudaError_t prepare_decode_kernel<128, 1, 0, 1, 1>(int, uint32_t, int *);
template cudaError_t prepare_decode_kernel<128, 1, 1, 1, 1>(int, uint32_t, int *);
template cudaError_t prepare_decode_kernel<32, 1, 0, 1, 1>(int, uint32_t, int *);
template cudaError_t prepare_decode_kernel<32, 1, 1, 1, 1>(int, uint32_t, int *);
template cudaError_t prepare_decode_kernel<32, 3, 0, 1, 1>(int, uint32_t, int *);
template cudaError_t prepare_decode_kernel<32, 3, 1, 1, 1>(int, uint32_t, int *);
template cudaError_t prepare_decode_kernel<64, 1, 0, 1, 1>(int, uint32_t, int *);
template cudaError_t prepare_decode_kernel<64, 1, 1, 1, 1>(int, uint32_t, int *);

}  // namespace aecct
