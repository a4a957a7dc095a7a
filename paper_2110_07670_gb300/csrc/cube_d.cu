// cube_d.cu -- compile-time pass kernels for the N^3 boxes N = 36, 40, 48, 50.
#include "pass_kernel.cuh"
#include "plane.cuh"
#include "zline.cuh"

namespace ace {

template cudaError_t pass_detail::dispatch_cube<36>(const PassArgs&, const PassShape&, int, int, int, int, int,
                                                  cudaStream_t);
template cudaError_t zline_launch<36>(const PassArgs&, int, cudaStream_t);
template cudaError_t tplane_launch<36>(int, const PassArgs&, int, cudaStream_t);
template cudaError_t pass_detail::dispatch_cube<40>(const PassArgs&, const PassShape&, int, int, int, int, int,
                                                  cudaStream_t);
template cudaError_t zline_launch<40>(const PassArgs&, int, cudaStream_t);
template cudaError_t tplane_launch<40>(int, const PassArgs&, int, cudaStream_t);
template cudaError_t pass_detail::dispatch_cube<48>(const PassArgs&, const PassShape&, int, int, int, int, int,
                                                  cudaStream_t);
template cudaError_t zline_launch<48>(const PassArgs&, int, cudaStream_t);
template cudaError_t tplane_launch<48>(int, const PassArgs&, int, cudaStream_t);
template cudaError_t pass_detail::dispatch_cube<50>(const PassArgs&, const PassShape&, int, int, int, int, int,
                                                  cudaStream_t);
template cudaError_t zline_launch<50>(const PassArgs&, int, cudaStream_t);
template cudaError_t tplane_launch<50>(int, const PassArgs&, int, cudaStream_t);

}  // namespace ace
