// cube_e.cu -- compile-time pass kernels for the N^3 boxes N = 54, 64, 72.
#include "pass_kernel.cuh"
#include "plane.cuh"
#include "zline.cuh"

namespace ace {

template cudaError_t pass_detail::dispatch_cube<54>(const PassArgs&, const PassShape&, int, int, int, int, int,
                                                  cudaStream_t);
template cudaError_t zline_launch<54>(const PassArgs&, int, cudaStream_t);
template cudaError_t tplane_launch<54>(int, const PassArgs&, int, cudaStream_t);
template cudaError_t pass_detail::dispatch_cube<64>(const PassArgs&, const PassShape&, int, int, int, int, int,
                                                  cudaStream_t);
template cudaError_t zline_launch<64>(const PassArgs&, int, cudaStream_t);
template cudaError_t tplane_launch<64>(int, const PassArgs&, int, cudaStream_t);
template cudaError_t pass_detail::dispatch_cube<72>(const PassArgs&, const PassShape&, int, int, int, int, int,
                                                  cudaStream_t);
template cudaError_t zline_launch<72>(const PassArgs&, int, cudaStream_t);
template cudaError_t tplane_launch<72>(int, const PassArgs&, int, cudaStream_t);

}  // namespace ace
