// cube_f.cu -- compile-time pass kernels for the N^3 boxes N = 128, 144.
#include "pass_kernel.cuh"
#include "plane.cuh"
#include "zline.cuh"

namespace ace {

template cudaError_t pass_detail::dispatch_cube<128>(const PassArgs&, const PassShape&, int, int, int, int, int,
                                                  cudaStream_t);
template cudaError_t zline_launch<128>(const PassArgs&, int, cudaStream_t);
template cudaError_t tplane_launch<128>(int, const PassArgs&, int, cudaStream_t);
template cudaError_t pass_detail::dispatch_cube<144>(const PassArgs&, const PassShape&, int, int, int, int, int,
                                                  cudaStream_t);
template cudaError_t zline_launch<144>(const PassArgs&, int, cudaStream_t);
template cudaError_t tplane_launch<144>(int, const PassArgs&, int, cudaStream_t);

}  // namespace ace
