// generic.cu -- launchers of the single-precision passes on runtime-size boxes.
#include "generic.cuh"

#include <algorithm>

namespace ace {

using namespace generic_detail;

namespace {

size_t plane_smem(int n1, int n2) { return ((size_t)n1 * (n2 | 1) + n1 + n2) * sizeof(cx<float>); }
size_t pencil_smem(int n0) { return (size_t)n0 * (128 + sizeof(cx<float>)); }

// Threads of a plane block: about 24 warps per SM over the blocks whose tiles
// the shared memory holds, no more than the plane's butterflies of radix 8.
int plane_threads(int n1, int n2) {
    const int blocks = std::max(1, (int)((228 * 1024) / (plane_smem(n1, n2) + 2048)));
    int nt = (kPlaneThreads / blocks + 31) / 32 * 32;
    nt = std::min(nt, (n1 * n2 / 8 + 31) / 32 * 32);
    return std::min(std::max(nt, 128), kPlaneThreads);
}

// The largest dynamic shared memory of a kernel here: the device's limit for a
// block less the kernel's static part.
int smem_max() {
    int dev = 0, lim = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        cudaGetLastError();
    return (lim > 0 ? lim : 227 * 1024) - 1024;
}

template <void (*k)(PassArgs)>
cudaError_t launch_planes(const PassArgs& a, int batch, cudaStream_t st) {
    static std::atomic<unsigned long long> done{0};
    const size_t smem = plane_smem(a.n1, a.n2);
    cudaError_t e = kernel_limits((const void*)k, smem_max(), true, done);
    if (e != cudaSuccess) return e;
    k<<<dim3((unsigned)a.n0, (unsigned)batch), plane_threads(a.n1, a.n2), smem, st>>>(a);
    return cudaGetLastError();
}

template <typename V, int MODE>
cudaError_t launch_pencils(const PassArgs& a, int batch, cudaStream_t st) {
    const int units = a.n1 * a.n2 / (int)(sizeof(V) / 4);
    static std::atomic<unsigned long long> done{0};
    const size_t smem = pencil_smem(a.n0);
    cudaError_t e = kernel_limits((const void*)pencils<V, MODE>, smem_max(), true, done);
    if (e != cudaSuccess) return e;
    const int U = Units<V>::U;
    pencils<V, MODE><<<dim3((unsigned)((units + U - 1) / U), (unsigned)batch), 32, smem, st>>>(a, units);
    return cudaGetLastError();
}

template <typename V, bool INVERSE>
cudaError_t launch_sphere(const PassArgs& a, const SphereArgs& sp, int batch, cudaStream_t st) {
    static std::atomic<unsigned long long> done{0};
    const int units = a.n1 * a.n2 / (int)(sizeof(V) / 4), U = Units<V>::U;
    const size_t smem = pencil_smem(a.n0);
    const auto k = INVERSE ? sphere_inverse<V> : sphere_forward<V>;
    cudaError_t e = kernel_limits((const void*)k, smem_max(), true, done);
    if (e != cudaSuccess) return e;
    const int items = INVERSE ? units : sp.nlist;
    k<<<dim3((unsigned)((items + U - 1) / U), (unsigned)batch), 32, smem, st>>>(a, units, sp);
    return cudaGetLastError();
}

}  // namespace

bool generic_supported(int n0, int n1, int n2) {
    const size_t smem_limit = (size_t)smem_max();
    return n0 >= 2 && n1 >= 2 && n2 >= 2 && plane_smem(n1, n2) <= smem_limit && pencil_smem(n0) <= smem_limit;
}

cudaError_t generic_plane_launch(const PassArgs& a, int pro, int epi, int batch, cudaStream_t st) {
    if (epi == EPI_STORE)
        return pro == PRO_PAIR ? launch_planes<plane_forward<PRO_PAIR>>(a, batch, st)
                               : launch_planes<plane_forward<PRO_PACK2>>(a, batch, st);
    return epi == EPI_ACCUM ? launch_planes<plane_inverse<EPI_ACCUM>>(a, batch, st)
                            : launch_planes<plane_inverse<EPI_SPLIT>>(a, batch, st);
}

cudaError_t generic_pencil_launch(const PassArgs& a, int mode, int batch, cudaStream_t st) {
    // pairs of pencils where a z row holds an even count (units stay 16-byte aligned)
    if ((long long)a.n1 * a.n2 % 2 == 0) {
        if (mode == 0) return launch_pencils<f2, 0>(a, batch, st);
        return mode < 0 ? launch_pencils<f2, -1>(a, batch, st) : launch_pencils<f2, +1>(a, batch, st);
    }
    if (mode == 0) return launch_pencils<float, 0>(a, batch, st);
    return mode < 0 ? launch_pencils<float, -1>(a, batch, st) : launch_pencils<float, +1>(a, batch, st);
}

int sphere_unit(int n1, int n2) { return (long long)n1 * n2 % 2 == 0 ? 2 : 1; }

cudaError_t sphere_launch(const PassArgs& a, const SphereArgs& sp, bool inverse, int batch, cudaStream_t st) {
    if (sphere_unit(a.n1, a.n2) == 2)
        return inverse ? launch_sphere<f2, true>(a, sp, batch, st) : launch_sphere<f2, false>(a, sp, batch, st);
    return inverse ? launch_sphere<float, true>(a, sp, batch, st) : launch_sphere<float, false>(a, sp, batch, st);
}

}  // namespace ace
