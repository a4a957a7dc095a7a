// zline.cuh -- the Coulomb pass of the pair Poisson solves (Eq. 3) on the
// compile-time N^3 boxes: forward FFT along z, times the Coulomb kernel
// 4 pi / |G|^2 / N (G = 0 dropped), inverse FFT along z.
//
// Two forms: the pass's own kernel zline_coulomb (below, pencils in pairs,
// packed arithmetic), and pencils_compute, the persistent pipeline's
// (pipeline.cuh), where every z line belongs to two lanes of one warp (lanes l
// and l + 16) and a warp owns G <= 16 consecutive pencils of the plane.  Both
// split a line's butterflies over lanes, so stages need only __syncwarp and no
// block-wide barrier exists, and touch whole 128-byte runs at every step.
//
// Per pencil the stages are: forward stages 0 .. S-2 in shared memory; the
// last forward stage, the Coulomb factors and the first inverse stage fused
// in registers (they act on the same butterflies); inverse stages S-2 .. 1 in
// shared memory; inverse stage 0 from shared memory straight to global memory.
// The Coulomb factors come from a table in the spectrum's own layout
// (digit-reversed z position, then the plane's stored slot), read once per
// element; the pass itself never needs to know the plane layout.
#pragma once

#include "fft_core.cuh"
#include "internal.h"
#include "tma.cuh"

namespace ace {
namespace zline_detail {

// Stage of the forward (SGN < 0) or inverse (SGN > 0) transform on one pencil
// held in shared memory with element stride G.
template <int RAD, int SGN, int N, int LB, int G>
__device__ __forceinline__ void pencil_stage(cx<float>* col, const cx<float>* tw, int h) {
    constexpr int M = LB / RAD, NB = N / RAD, TS = N / LB;
#pragma unroll 2
    for (int i = h; i < NB; i += 2) {
        const int beta = i / M, j = i - beta * M;
        butterfly_core<RAD, SGN, float>(col + (beta * LB + j) * G, M * G, tw, TS * j, M > 1 && j > 0);
    }
}

// Last forward stage (blocks of RAD adjacent positions, no twiddles), the
// Coulomb factors, and the first inverse stage on the same RAD positions.
template <int RAD, int N, int G>
__device__ __forceinline__ void pencil_middle(cx<float>* col, const float* krow, int h) {
    constexpr int NB = N / RAD;
    constexpr long long NN = (long long)N * N;
#pragma unroll 2
    for (int beta = h; beta < NB; beta += 2) {
        float k[RAD];
        cx<float> u[RAD];
#pragma unroll
        for (int q = 0; q < RAD; ++q) k[q] = __ldg(krow + (beta * RAD + q) * NN);
#pragma unroll
        for (int q = 0; q < RAD; ++q) u[q] = col[(beta * RAD + q) * G];
        Dft<RAD, -1, float>::run(u);
#pragma unroll
        for (int q = 0; q < RAD; ++q) u[q] = scale(u[q], k[q]);
        Dft<RAD, +1, float>::run(u);
#pragma unroll
        for (int q = 0; q < RAD; ++q) col[(beta * RAD + q) * G] = u[q];
    }
}

// Inverse stage 0 (blocks of the whole line): conjugate twiddles, butterfly,
// and the results in natural order straight to global memory (stride N^2).
template <int RAD, int N, int G>
__device__ __forceinline__ void pencil_last(const cx<float>* col, const cx<float>* tw, cx<float>* out, int h) {
    constexpr int M = N / RAD;
    constexpr long long NN = (long long)N * N;
#pragma unroll 2
    for (int j = h; j < M; j += 2) {
        cx<float> u[RAD];
#pragma unroll
        for (int q = 0; q < RAD; ++q) u[q] = col[(j + q * M) * G];
        if (j > 0) {
#pragma unroll
            for (int q = 1; q < RAD; ++q) {
                cx<float> w = tw[q * j];
                w.im = -w.im;
                u[q] = cmul(u[q], w);
            }
        }
        Dft<RAD, +1, float>::run(u);
#pragma unroll
        for (int s = 0; s < RAD; ++s) out[(j + s * M) * NN] = u[s];
    }
}

// The transforms of one group of G pencils held in buf ([N][G], element
// stride G), by one warp: forward stages, the fused middle with the Coulomb
// factors kern_p0[z N^2 + p], the inverse stages, and the results to
// dst_p0[z N^2 + p] (p = 0 .. G-1, in natural z order).
template <int N, int G, int F0 = 0>
__device__ __forceinline__ void pencils_compute(cx<float>* buf, const cx<float>* tw, const float* kern_p0,
                                                cx<float>* dst_p0, int lane) {
    using PL = CPlan<N, F0>;
    // lanes past the group's pencils (G < 16) skip every step but the syncs
    const int pl = lane & 15, h = lane >> 4;
    const bool on = pl < G;
    cx<float>* col = buf + pl;
    CLoop<0, PL::stages - 1>::run([&](auto sc) {
        constexpr int s = decltype(sc)::value;
        if (on) pencil_stage<PL::radix(s), -1, N, PL::block_len(s), G>(col, tw, h);
        __syncwarp();
    });
    if (on) pencil_middle<PL::radix(PL::stages - 1), N, G>(col, kern_p0 + pl, h);
    __syncwarp();
    CLoop<0, PL::stages - 2>::run([&](auto sc) {
        constexpr int s = PL::stages - 2 - decltype(sc)::value;
        if (on) pencil_stage<PL::radix(s), +1, N, PL::block_len(s), G>(col, tw, h);
        __syncwarp();
    });
    cx<float>* out = dst_p0 + pl;
    if (on) pencil_last<PL::radix(0), N, G>(col, tw, out, h);
}

// ---------------------------------------------------------------- the pass
// Packed form (f2): pencils p and p + 1, neighbours in the plane's layout, run
// through every butterfly together, one packed instruction doing the work of
// two.  A warp owns 8 pencil pairs (128 bytes of every z row, copied by 16-byte
// cp.async; four lanes share a pair's butterflies), a block is one warp.  A
// pair's 16 bytes {re0, im0, re1, im1} become {re0, re1}, {im0, im1} in the
// first stage's registers and turn back in the last's.
// Bound: DRAM (0.85 GB per 64 transforms of 96^3 at 5.6 TB/s) with the shared
// memory pipe at 68%.  Measured per 64 / 38 / 16 transforms of 96^3 / 120^3 /
// 160^3: 153 / 191 / 233 us, where single pencils on two lanes each, fetched by
// one 128-byte bulk copy per z row (some 8 instructions each: a lane's copies
// are issued one by one), took 179 / 266 / 316.  Fully unrolled rounds (more
// registers, more code) and persistent warps that fetch the next group behind
// the last stage are slower (96^3 165 and 154 us).

constexpr int kPairsPerWarp = 8;

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ f2 ldg2(const float* p) {
    f2 r;
    r.v = __ldg(reinterpret_cast<const unsigned long long*>(p));
    return r;
}
// two neighbouring complex values <-> their real and imaginary parts paired
__device__ __forceinline__ cx<f2> swap_mid(cx<f2> a) {
    return mk(mk_f2(lo(a.re), lo(a.im)), mk_f2(hi(a.re), hi(a.im)));
}

// NAT: the padded natural planes of plane.cuh (pads ride along)
template <int N, int F0, bool NAT>
__global__ void __launch_bounds__(32) zline_coulomb(PassArgs a) {
    using PL = CPlan<N, F0>;
    using c2 = cx<f2>;
    static_assert(PL::stages == 2 && N % 2 == 0, "two stages, pencils in pairs");
    constexpr int U = kPairsPerWarp, L = 32 / U;
    constexpr int R0 = PL::radix(0), R1 = PL::radix(1), M0 = N / R0, B1 = N / R1;
    constexpr long long HU = (NAT ? plane_elems(N) : N * N) / 2;   // pencil pairs of the box
    constexpr long long ZU = (NAT ? plane_stride(N) : N * N) / 2;  // ... and from plane to plane
    extern __shared__ __align__(128) unsigned char smem_raw[];
    c2* buf = reinterpret_cast<c2*>(smem_raw);                  // [N][U]
    cx<float>* tw = reinterpret_cast<cx<float>*>(buf + N * U);  // [N]
    const int lane = threadIdx.x, l = lane % U, h = lane / U;
    const long long p = (long long)blockIdx.x * U + l;
    const int t = blockIdx.y;
    const bool on = HU % U == 0 || p < HU;  // lanes past the last pair only keep the barriers
    const c2* src = reinterpret_cast<const c2*>(reinterpret_cast<const cx<float>*>(a.src) + t * a.src_tstride) + p;
    if (on)
#pragma unroll 4
        for (int z = h; z < N; z += L) cp_async16(buf + z * U + l, src + z * ZU);
    for (int j = lane; j < N; j += 32) tw[j] = reinterpret_cast<const cx<float>*>(a.twz)[j];
    cp_async_wait();
    __syncwarp();
    c2* col = buf + l;
    if (on) {
#pragma unroll 1
        for (int j = h; j < M0; j += L) {
            c2 u[R0];
#pragma unroll
            for (int k = 0; k < R0; ++k) u[k] = swap_mid(col[(j + k * M0) * U]);
            Dft<R0, -1, f2>::run(u);
#pragma unroll
            for (int s = 1; s < R0; ++s) u[s] = cmul(u[s], tw[s * j]);
#pragma unroll
            for (int s = 0; s < R0; ++s) col[(j + s * M0) * U] = u[s];
        }
    }
    __syncwarp();
    if (on) {
        // last forward stage, the Coulomb factors and the first inverse stage
        // act on the same butterflies
        const float* kern = reinterpret_cast<const float*>(a.kern) + 2 * p;
#pragma unroll 1
        for (int b = h; b < B1; b += L) {
            f2 k[R1];
            c2 u[R1];
#pragma unroll
            for (int q = 0; q < R1; ++q) k[q] = ldg2(kern + (b * R1 + q) * (2 * ZU));
#pragma unroll
            for (int q = 0; q < R1; ++q) u[q] = col[(b * R1 + q) * U];
            Dft<R1, -1, f2>::run(u);
#pragma unroll
            for (int q = 0; q < R1; ++q) u[q] = scale(u[q], k[q]);
            Dft<R1, +1, f2>::run(u);
#pragma unroll
            for (int q = 0; q < R1; ++q) col[(b * R1 + q) * U] = u[q];
        }
    }
    __syncwarp();
    if (on) {
        c2* out = reinterpret_cast<c2*>(reinterpret_cast<cx<float>*>(a.dst) + t * a.dst_tstride) + p;
#pragma unroll 1
        for (int j = h; j < M0; j += L) {
            c2 u[R0];
            u[0] = col[j * U];
#pragma unroll
            for (int q = 1; q < R0; ++q) {
                cx<float> w = tw[q * j];
                w.im = -w.im;
                u[q] = cmul(col[(j + q * M0) * U], w);
            }
            Dft<R0, +1, f2>::run(u);
#pragma unroll
            for (int s = 0; s < R0; ++s) out[(j + s * M0) * ZU] = swap_mid(u[s]);
        }
    }
}

}  // namespace zline_detail

template <int N, int F0, bool NAT>
cudaError_t zline_launch_nat(const PassArgs& a, int batch, cudaStream_t st) {
    constexpr int U = zline_detail::kPairsPerWarp;
    auto k = zline_detail::zline_coulomb<N, F0, NAT>;
    const size_t smem = (size_t)N * U * sizeof(cx<f2>) + N * sizeof(cx<float>);
    static std::atomic<unsigned long long> done{0};
    cudaError_t e = kernel_limits((const void*)k, (int)smem, true, done);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)(((NAT ? plane_elems(N) : N * N) / 2 + U - 1) / U), (unsigned)batch);
    k<<<grid, 32, smem, st>>>(a);
    return cudaGetLastError();
}

// F0: the first radix of the z axis (0: make_axis_plan's choice)
template <int N, int F0 = 0>
cudaError_t zline_launch(const PassArgs& a, int batch, cudaStream_t st) {
    return a.natural ? zline_launch_nat<N, F0, true>(a, batch, st) : zline_launch_nat<N, F0, false>(a, batch, st);
}

}  // namespace ace
