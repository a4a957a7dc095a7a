// plane.cuh -- the two plane passes of the pair Poisson solves (Eq. 2-4) on
// the compile-time N^3 boxes, with thread-owned lines:
//
//   forward  (pair_fwd):   rho = phi_a phi_b + i phi_c phi_d on plane z, 2-D
//                          forward FFT, spectrum plane stored;
//   inverse  (inv_accum, inv_accum_natural):  2-D inverse FFT of a spectrum
//                          plane, then W_a += v phi_b, W_b += v phi_a, ... and
//                          the pair energies sum rho v (Eq. 4).
//
// Between the passes (and through the per-pencil Coulomb pass) a spectrum
// plane has one of two layouts (positions digit-reversed after the forward
// stages in both):
//   natural (the hybrid variant): the shared tile as it stands, pads included,
//     so that a plane is one bulk copy each way;
//   transposed: [x][y].  The pass that works on x lines reads or writes global
//     memory straight from its butterflies with the lanes along y.
// Either way the pass that works on y lines meets the real-space functions
// with the lanes along x, whole 128-byte lines.
//
// Every line (a y column or an x row of the plane) belongs to two to four
// threads (plane_tpl), thread l, N + l, ..., which split its butterflies; a
// warp's lanes take 32 consecutive lines, and a line's threads meet at block
// barriers between the stages.  The rows of the shared tile are padded so that
// 16 lanes on 16 consecutive rows, or on 16 consecutive columns, hit 16
// distinct bank pairs (plane_row).  The accumulation after the inverse runs on
// 4-wide vectors from the tile.  Both axes have two stages (radix R0 with
// N / R0 butterflies of stride N / R0, then radix R1 on adjacent positions).
//
// Bound: the shared memory / L1 pipe and, between the phases of a block, its
// barriers, so resident blocks count.  Measured per 64 / 38 transforms of
// 96^3 / 120^3 (P1, P3, alone): 168, 224 / 269, 366 us.  Before the natural
// layout P1 wrote rows permuted for the tile kernels and those accumulated:
// 185, 234 / 314, 435; rows of N + 1 at 120^3 (one block per SM) 322, 449.
#pragma once

#include "fft_core.cuh"
#include "internal.h"
#include "tma.cuh"

namespace ace {
namespace plane_detail {

// F0: the first radix of both axes (0: make_axis_plan's choice); TPL: threads
// per line (2, or 4 for the large planes that leave one block per SM)
template <int N, int F0 = 0, int TPL = 2>
struct Geo {
    using PL = CPlan<N, F0>;
    static_assert(PL::stages == 2, "plane passes assume two stages per axis");
    static constexpr int R0 = PL::radix(0), R1 = PL::radix(1);
    static constexpr int M0 = N / R0;  // stage-0 butterflies per line (stride M0)
    static constexpr int B1 = N / R1;  // stage-1 butterflies per line (adjacent)
    static constexpr int NT = (TPL * N + 31) / 32 * 32;
    static constexpr bool HALF = plane_half_pad(N);
    static constexpr int E = plane_elems(N);
    static constexpr uint32_t kPlaneBytes = (uint32_t)(E * sizeof(cx<float>));
    // tile, twiddles (HALF: none, read from global memory), a barrier and a flag
    static constexpr size_t smem = (size_t)(E + (HALF ? 0 : N)) * sizeof(cx<float>) + 16;
    // resident blocks per SM: its shared memory, at most 32, and no more than
    // leave 72 registers per thread
    static constexpr int kSmemBlocks = plane_blocks((int)smem);
    static constexpr int kRegBlocks = 65536 / (NT * 72) > 0 ? 65536 / (NT * 72) : 1;
    static constexpr int kMinBlocks = kSmemBlocks < kRegBlocks ? kSmemBlocks : kRegBlocks;
    // start of row y, and of row y + dy: with HALF a constant from row y where
    // y or dy is even, as in both stages of a radix plan with M0 and R1 even
    static __device__ __forceinline__ int row(int y) { return plane_row(N, y); }
    static __device__ __forceinline__ int row(int y, int dy) {
        if constexpr (HALF && (M0 % 2 != 0 || R1 % 2 != 0)) return plane_row(N, y + dy);
        return plane_row(N, y) + dy * N + (HALF ? dy >> 1 : dy);
    }
};

// the N twiddles: copied behind the tile, or (HALF) as they are in global memory
template <class G>
__device__ __forceinline__ const cx<float>* twiddles(const PassArgs& a, cx<float>* tile) {
    const cx<float>* g = reinterpret_cast<const cx<float>*>(a.twx);
    if constexpr (G::HALF) {
        return g;
    } else {
        cx<float>* tw = tile + G::E;
        for (int j = threadIdx.x; j < G::M0 * G::R0; j += G::NT) tw[j] = g[j];
        return tw;
    }
}

// forward stage-0 twiddles on the outputs (DIF), inverse on the inputs (conjugate)
template <int R>
__device__ __forceinline__ void tw_out(cx<float> (&u)[R], const cx<float>* tw, int j) {
    if (j > 0) {
#pragma unroll
        for (int s = 1; s < R; ++s) u[s] = cmul(u[s], tw[s * j]);
    }
}
template <int R>
__device__ __forceinline__ void tw_in_conj(cx<float> (&u)[R], const cx<float>* tw, int j) {
    if (j > 0) {
#pragma unroll
        for (int q = 1; q < R; ++q) {
            cx<float> w = tw[q * j];
            w.im = -w.im;
            u[q] = cmul(u[q], w);
        }
    }
}

// threads per line by how many plane blocks an SM's shared memory holds:
// fewer blocks, more warps per block (2 / 3 / 4 threads: P1 + P3 of 64
// transforms of 96^3, three blocks, 392 / 389 / 531 us; of 38 of 100^3, two,
// 359 / 341 / 345 us; at one block 5 threads are 0-5% slower than 4)
template <int N>
constexpr int plane_tpl() {
    constexpr int blocks = Geo<N, 0, 2>::kSmemBlocks;
    return blocks >= 3 ? 2 : blocks == 2 ? 3 : 4;
}

__device__ __forceinline__ float4 ldg4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 mul4(float4 a, float4 b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }
__device__ __forceinline__ float4 fma4(float4 a, float4 b, float4 c) {
    return make_float4(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y), fmaf(a.z, b.z, c.z), fmaf(a.w, b.w, c.w));
}
__device__ __forceinline__ float dot4(float4 a, float4 b) { return a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w; }
__device__ __forceinline__ void red_add4(float* p, float4 v) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

// 8-byte global -> shared asynchronous copy (completes at cp_async_wait_all)
__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gsrc) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Pull the plane-z slices of transform tt's functions (and accumulators) into L2.
__device__ __forceinline__ void prefetch_planes(const PassArgs& a, const Quad& q, long long off, uint32_t bytes,
                                                long long N3, bool with_w) {
    const float* fl = reinterpret_cast<const float*>(a.fl);
    const float* fr = reinterpret_cast<const float*>(a.fr);
    prefetch_l2(fl + q.a * N3 + off, bytes);
    prefetch_l2(fr + q.b * N3 + off, bytes);
    if (q.c >= 0) {
        if (q.c != q.a) prefetch_l2(fl + q.c * N3 + off, bytes);
        prefetch_l2(fr + q.d * N3 + off, bytes);
    }
    if (with_w) {
        const float* wl = reinterpret_cast<const float*>(a.accl);
        prefetch_l2(wl + q.a * N3 + off, bytes);
        if (q.c >= 0 && q.c != q.a) prefetch_l2(wl + q.c * N3 + off, bytes);
        if (a.symmetric) {
            const float* wr = reinterpret_cast<const float*>(a.accr);
            if (q.b != q.a) prefetch_l2(wr + q.b * N3 + off, bytes);
            if (q.c >= 0 && q.d != q.c) prefetch_l2(wr + q.d * N3 + off, bytes);
        }
    }
}

// Plane z of one transform (quad q): pair product, 2-D forward FFT, and the
// plane stored into spec_t (the transform's spectrum) transposed ([x][y]), or
// with NATURAL left in the tile (row y, x position p at row(y) + p) for the
// caller to store after a barrier.
// tw holds the N twiddles in shared memory (visible to the block); the
// block's threads all call this.
template <int N, bool NATURAL = false, int F0 = 0, int TPL = 2>
__device__ __forceinline__ void pair_fwd_plane(const PassArgs& a, const Quad& q, int z, cx<float>* tile,
                                               const cx<float>* tw, cx<float>* spec_t) {
    using G = Geo<N, F0, TPL>;
    constexpr long long NN = (long long)N * N, N3 = NN * N;
    const long long plane0 = (long long)z * NN;
    const int h = (int)threadIdx.x / N, line = (int)threadIdx.x - h * N;
    const bool active = h < TPL;  // threads past TPL N idle
    const bool has2 = q.c >= 0;

    // y lines (thread owns column x): stage 0 straight from the functions
    if (active) {
        const int x = line;
        const float* pa = reinterpret_cast<const float*>(a.fl) + q.a * N3 + plane0 + x;
        const float* pb = reinterpret_cast<const float*>(a.fr) + q.b * N3 + plane0 + x;
        const float* pc = reinterpret_cast<const float*>(a.fl) + (has2 ? q.c : q.a) * N3 + plane0 + x;
        const float* pd = reinterpret_cast<const float*>(a.fr) + (has2 ? q.d : q.b) * N3 + plane0 + x;
        for (int j = h; j < G::M0; j += TPL) {
            cx<float> u[G::R0];
#pragma unroll
            for (int k = 0; k < G::R0; ++k) {
                const long long r = (long long)(j + k * G::M0) * N;
                u[k].re = __ldg(pa + r) * __ldg(pb + r);
                u[k].im = has2 ? __ldg(pc + r) * __ldg(pd + r) : 0.0f;
            }
            Dft<G::R0, -1, float>::run(u);
            tw_out<G::R0>(u, tw, j);
#pragma unroll
            for (int s = 0; s < G::R0; ++s) tile[G::row(j, s * G::M0) + x] = u[s];
        }
    }
    __syncthreads();
    if (active) {
        const int x = line;
        for (int b = h; b < G::B1; b += TPL) {
            cx<float> u[G::R1];
#pragma unroll
            for (int k = 0; k < G::R1; ++k) u[k] = tile[G::row(b * G::R1, k) + x];
            Dft<G::R1, -1, float>::run(u);
#pragma unroll
            for (int s = 0; s < G::R1; ++s) tile[G::row(b * G::R1, s) + x] = u[s];
        }
    }
    __syncthreads();

    // x lines (thread owns row y): stage 0 in shared memory, stage 1 to the
    // transposed spectrum plane
    if (active) {
        cx<float>* row = tile + G::row(line);
        for (int j = h; j < G::M0; j += TPL) {
            cx<float> u[G::R0];
#pragma unroll
            for (int k = 0; k < G::R0; ++k) u[k] = row[j + k * G::M0];
            Dft<G::R0, -1, float>::run(u);
            tw_out<G::R0>(u, tw, j);
#pragma unroll
            for (int s = 0; s < G::R0; ++s) row[j + s * G::M0] = u[s];
        }
    }
    __syncthreads();
    if (active) {
        cx<float>* row = tile + G::row(line);
        cx<float>* out = spec_t + plane0 + line;
        for (int b = h; b < G::B1; b += TPL) {
            cx<float> u[G::R1];
#pragma unroll
            for (int k = 0; k < G::R1; ++k) u[k] = row[b * G::R1 + k];
            Dft<G::R1, -1, float>::run(u);
            if constexpr (NATURAL) {
#pragma unroll
                for (int s = 0; s < G::R1; ++s) row[b * G::R1 + s] = u[s];
            } else {
#pragma unroll
                for (int s = 0; s < G::R1; ++s) out[(long long)(b * G::R1 + s) * N] = u[s];
            }
        }
    }
}

template <int N, bool NATURAL, int F0, int TPL>
__global__ void __launch_bounds__(Geo<N, F0, TPL>::NT, Geo<N, F0, TPL>::kMinBlocks) pair_fwd(PassArgs a) {
    using G = Geo<N, F0, TPL>;
    constexpr long long NN = (long long)N * N, N3 = NN * N;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    cx<float>* tile = reinterpret_cast<cx<float>*>(smem_raw);  // (y, x) at row(y) + x
    const cx<float>* tw = twiddles<G>(a, tile);
    const int z = blockIdx.x, t = blockIdx.y;
    const Quad q = a.quads[a.t0 + t];
    const long long plane0 = (long long)z * NN;
    if (threadIdx.x == 32 && a.lookahead > 0 && t + a.lookahead < (int)gridDim.y && (NN * 4) % 16 == 0)
        prefetch_planes(a, a.quads[a.t0 + t + a.lookahead], plane0, (uint32_t)(NN * 4), N3, false);
    if constexpr (NATURAL)  // the pads go out with the plane
        for (int y = threadIdx.x; y < N; y += G::NT)
            if (!G::HALF || y % 2 != 0) tile[G::row(y) + N] = mk(0.0f, 0.0f);
    __syncthreads();
    cx<float>* dst = reinterpret_cast<cx<float>*>(a.dst) + t * a.dst_tstride;
    pair_fwd_plane<N, NATURAL, F0, TPL>(a, q, z, tile, tw, dst);
    if constexpr (NATURAL) {
        // the tile as it stands is the plane: one bulk store (64 transforms
        // of 96^3: 168 us, 185 with the tile's swizzled rows written out by the
        // threads, 190 with 16-byte stores of this layout; equal where one
        // block fills the SM)
        fence_proxy_async_smem();
        __syncthreads();
        if (threadIdx.x == 0) {
            bulk_store(dst + (long long)z * plane_stride(N), tile, G::kPlaneBytes);
            bulk_commit();
            bulk_wait_read_all();
        }
    }
}

// Inputs of the inverse pass: thread (row y, half h) needs the transposed
// plane's x positions of its first butterflies in its row of the tile.
// Asynchronous 8-byte copies (the standalone kernel: all in flight at once,
// completed by cp_async_wait_all) ...
template <int N, int F0 = 0, int TPL = 2>
__device__ __forceinline__ void inv_issue_copies(const cx<float>* plane_in, cx<float>* tile) {
    using G = Geo<N, F0, TPL>;
    const int h = (int)threadIdx.x / N, line = (int)threadIdx.x - h * N;
    if (h < TPL) {
        const cx<float>* in = plane_in + line;
        cx<float>* row = tile + G::row(line);
        for (int b = h; b < G::B1; b += TPL)
#pragma unroll
            for (int k = 0; k < G::R1; ++k) cp_async8(row + b * G::R1 + k, in + (long long)(b * G::R1 + k) * N);
    }
    cp_async_commit();
}

// ... or loads that bypass L1 (ld.global.cg), for spectra written by other
// blocks of the same kernel.
__device__ __forceinline__ cx<float> ld_cg2(const cx<float>* p) {
    float2 v;
    asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return mk(v.x, v.y);
}
template <int N, int F0 = 0, int TPL = 2>
__device__ __forceinline__ void inv_load_cg(const cx<float>* plane_in, cx<float>* tile) {
    using G = Geo<N, F0, TPL>;
    const int h = (int)threadIdx.x / N, line = (int)threadIdx.x - h * N;
    if (h < TPL) {
        const cx<float>* in = plane_in + line;
        cx<float>* row = tile + G::row(line);
        for (int b = h; b < G::B1; b += TPL) {
            cx<float> u[G::R1];
#pragma unroll
            for (int k = 0; k < G::R1; ++k) u[k] = ld_cg2(in + (long long)(b * G::R1 + k) * N);
#pragma unroll
            for (int k = 0; k < G::R1; ++k) row[b * G::R1 + k] = u[k];
        }
    }
}

// Plane z of one transform (quad q), its inputs already in the tile (each
// thread's own): 2-D inverse FFT, then W_a += v phi_b, W_b += v phi_a, ...
// (Eq. 2) and the pair-energy partials (Eq. 4) into e_dst[2] (may be null).
// red: 2 * NT / 32 doubles of shared memory, the tile's own if wished.  Every thread of the block calls it.
template <int N, int F0 = 0, int TPL = 2>
__device__ __forceinline__ void inv_accum_plane(const PassArgs& a, const Quad& q, int z, cx<float>* tile,
                                                const cx<float>* tw, double* red, double* e_dst) {
    using G = Geo<N, F0, TPL>;
    static_assert(N % 2 == 0, "the epilogue's 4-wide vectors cross rows between two pairs only");
    constexpr long long NN = (long long)N * N, N3 = NN * N;
    const long long plane0 = (long long)z * NN;
    const int h = (int)threadIdx.x / N, line = (int)threadIdx.x - h * N;
    const bool active = h < TPL;  // threads past TPL N idle
    // x lines (thread owns row y): both inverse stages in shared memory
    if (active) {
        cx<float>* row = tile + G::row(line);
        for (int b = h; b < G::B1; b += TPL) {
            cx<float> u[G::R1];
#pragma unroll
            for (int k = 0; k < G::R1; ++k) u[k] = row[b * G::R1 + k];
            Dft<G::R1, +1, float>::run(u);
#pragma unroll
            for (int s = 0; s < G::R1; ++s) row[b * G::R1 + s] = u[s];
        }
    }
    __syncthreads();
    if (active) {
        cx<float>* row = tile + G::row(line);
        for (int j = h; j < G::M0; j += TPL) {
            cx<float> u[G::R0];
#pragma unroll
            for (int k = 0; k < G::R0; ++k) u[k] = row[j + k * G::M0];
            tw_in_conj<G::R0>(u, tw, j);
            Dft<G::R0, +1, float>::run(u);
#pragma unroll
            for (int s = 0; s < G::R0; ++s) row[j + s * G::M0] = u[s];
        }
    }
    __syncthreads();

    // y lines (thread owns column x): both inverse stages in shared memory
    if (active) {
        const int x = line;
        for (int b = h; b < G::B1; b += TPL) {
            cx<float> u[G::R1];
#pragma unroll
            for (int k = 0; k < G::R1; ++k) u[k] = tile[G::row(b * G::R1, k) + x];
            Dft<G::R1, +1, float>::run(u);
#pragma unroll
            for (int s = 0; s < G::R1; ++s) tile[G::row(b * G::R1, s) + x] = u[s];
        }
    }
    __syncthreads();
    if (active) {
        const int x = line;
        for (int j = h; j < G::M0; j += TPL) {
            cx<float> u[G::R0];
#pragma unroll
            for (int k = 0; k < G::R0; ++k) u[k] = tile[G::row(j, k * G::M0) + x];
            tw_in_conj<G::R0>(u, tw, j);
            Dft<G::R0, +1, float>::run(u);
#pragma unroll
            for (int s = 0; s < G::R0; ++s) tile[G::row(j, s * G::M0) + x] = u[s];
        }
    }
    __syncthreads();

    // Exchange accumulation (Eq. 2) and pair energies (Eq. 4) in 4-wide
    // vectors, consecutive lanes on consecutive vectors of the plane: every
    // load and every reduction covers whole 128-byte lines.  (Tasks of 4 rows
    // x 16 columns per half-warp, half lines each, took 315 against 224 us per
    // 64 transforms of 96^3, 119 against 103 at 72^3.)  N % 32 == 0: the 16
    // lanes of a half-warp take 2 rows x 32 columns, and the odd pitch separates
    // the rows' banks: one rotation step instead of tile_read4's two.
    float e1 = 0.0f, e2 = 0.0f;
    {
        const bool has2 = q.c >= 0, share = has2 && q.c == q.a, sym = a.symmetric != 0;
        const bool upd_b = sym && q.a != q.b, upd_d = sym && has2 && q.c != q.d;
        const float* la_p = reinterpret_cast<const float*>(a.fl) + q.a * N3 + plane0;
        const float* rb_p = reinterpret_cast<const float*>(a.fr) + q.b * N3 + plane0;
        const float* lc_p = reinterpret_cast<const float*>(a.fl) + (has2 ? q.c : q.a) * N3 + plane0;
        const float* rd_p = reinterpret_cast<const float*>(a.fr) + (has2 ? q.d : q.b) * N3 + plane0;
        float* wa_p = reinterpret_cast<float*>(a.accl) + q.a * N3 + plane0;
        float* wc_p = reinterpret_cast<float*>(a.accl) + (has2 ? q.c : q.a) * N3 + plane0;
        float* wb_p = sym ? reinterpret_cast<float*>(a.accr) + q.b * N3 + plane0 : nullptr;
        float* wd_p = sym ? reinterpret_cast<float*>(a.accr) + (has2 ? q.d : q.b) * N3 + plane0 : nullptr;
        constexpr bool TWO_ROWS = N % 32 == 0;
        // N^2 / 4 vectors over NT threads, taken U at a time with every load
        // issued before the first update
        constexpr int NTASK = N * N / 4, PER = (NTASK + G::NT - 1) / G::NT, U = PER == 1 ? 1 : 2;
        constexpr bool EVEN = PER % U == 0 && NTASK % G::NT == 0;
        const bool odd4 = threadIdx.x & 4;
        for (int k0 = 0; k0 < PER; k0 += U) {
            float4 la[U], rb[U], lc[U], rd[U];
            int rof[U], s01[U], s23[U];  // offsets in the plane; of elements 0, 1 and 2, 3 in the tile
            bool on[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int task = (int)threadIdx.x + (k0 + u) * G::NT;
                on[u] = EVEN || task < NTASK;
                if (!on[u]) continue;
                if constexpr (TWO_ROWS) {
                    const int grp = task >> 4, y = grp / (N / 32) * 2 + (task >> 3 & 1);
                    const int x = grp % (N / 32) * 32 + 4 * (task & 7);
                    rof[u] = y * N + x;
                    s01[u] = G::row(y) + x;
                    s23[u] = s01[u] + 2;
                } else {
                    rof[u] = 4 * task;
                    constexpr int PR = G::HALF ? 2 * N : N;  // elements between pads
                    s01[u] = rof[u] + rof[u] / PR;
                    s23[u] = N % 4 == 0 ? s01[u] + 2 : rof[u] + 2 + (rof[u] + 2) / PR;
                }
                la[u] = ldg4(la_p + rof[u]);
                rb[u] = ldg4(rb_p + rof[u]);
                if (has2) {
                    lc[u] = ldg4(lc_p + rof[u]);
                    rd[u] = ldg4(rd_p + rof[u]);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (!on[u]) continue;
                const int r = rof[u];
                cx<float> v[4];
                if constexpr (TWO_ROWS) {
                    const int p = odd4 ? s23[u] : s01[u], q2 = odd4 ? s01[u] : s23[u];
                    const cx<float> w0 = tile[p], w1 = tile[p + 1], w2 = tile[q2], w3 = tile[q2 + 1];
                    v[0] = odd4 ? w2 : w0;
                    v[1] = odd4 ? w3 : w1;
                    v[2] = odd4 ? w0 : w2;
                    v[3] = odd4 ? w1 : w3;
                } else {
                    tile_read4(tile, s01[u], s23[u], v);
                }
                const float4 v1 = make_float4(v[0].re, v[1].re, v[2].re, v[3].re);
                const float4 v2 = make_float4(v[0].im, v[1].im, v[2].im, v[3].im);
                float4 wa = mul4(v1, rb[u]);
                e1 += dot4(mul4(la[u], rb[u]), v1);
                if (has2) {
                    e2 += dot4(mul4(lc[u], rd[u]), v2);
                    if (share)
                        wa = fma4(v2, rd[u], wa);
                    else
                        red_add4(wc_p + r, mul4(v2, rd[u]));
                    if (upd_d) red_add4(wd_p + r, mul4(v2, lc[u]));
                }
                red_add4(wa_p + r, wa);
                if (upd_b) red_add4(wb_p + r, mul4(v1, la[u]));
            }
        }
    }
    if (e_dst != nullptr) {
        const double d1 = warp_sum_ff(e1), d2 = warp_sum_ff(e2);
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        __syncthreads();  // red may lie in the tile
        if (lane == 0) {
            red[2 * warp] = d1;
            red[2 * warp + 1] = d2;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double s1 = 0, s2 = 0;
            for (int w = 0; w < G::NT / 32; ++w) {
                s1 += red[2 * w];
                s2 += red[2 * w + 1];
            }
            e_dst[0] = s1;
            e_dst[1] = s2;
        }
    }
}

template <int N, int F0, int TPL>
__global__ void __launch_bounds__(Geo<N, F0, TPL>::NT, Geo<N, F0, TPL>::kMinBlocks) inv_accum(PassArgs a) {
    using G = Geo<N, F0, TPL>;
    constexpr long long NN = (long long)N * N, N3 = NN * N;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    cx<float>* tile = reinterpret_cast<cx<float>*>(smem_raw);
    const cx<float>* tw = twiddles<G>(a, tile);
    const int z = blockIdx.x, t = blockIdx.y;
    const long long plane0 = (long long)z * NN;
    inv_issue_copies<N, F0, TPL>(reinterpret_cast<const cx<float>*>(a.src) + t * a.src_tstride + plane0, tile);
    const Quad q = a.quads[a.t0 + t];
    // the accumulation reads up to four function planes and updates up to four
    // accumulator planes at the end: start pulling them into L2 now
    if (threadIdx.x == 32 && (NN * 4) % 16 == 0) prefetch_planes(a, q, plane0, (uint32_t)(NN * 4), N3, true);
    cp_async_wait_all();
    __syncthreads();
    inv_accum_plane<N, F0, TPL>(a, q, z, tile, tw, reinterpret_cast<double*>(tile),
                       a.e_part != nullptr ? a.e_part + ((long long)(a.t0 + t) * gridDim.x + z) * 2 : nullptr);
}

// The inverse pass from planes in the tile's own layout (the
// forward pass's NATURAL output): one bulk copy per plane.
template <int N, int F0, int TPL>
__global__ void __launch_bounds__(Geo<N, F0, TPL>::NT, Geo<N, F0, TPL>::kMinBlocks) inv_accum_natural(PassArgs a) {
    using G = Geo<N, F0, TPL>;
    constexpr long long NN = (long long)N * N, N3 = NN * N;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    cx<float>* tile = reinterpret_cast<cx<float>*>(smem_raw);
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + G::smem - 16);
    int* timed_out = reinterpret_cast<int*>(bar + 1);
    const int z = blockIdx.x, t = blockIdx.y;
    if (threadIdx.x == 0) {
        *timed_out = 0;
        mbar_init(bar, 1);
        fence_mbar_init();
        mbar_arrive_expect_tx(bar, G::kPlaneBytes);
        bulk_load(tile, reinterpret_cast<const cx<float>*>(a.src) + t * a.src_tstride + (long long)z * plane_stride(N),
                  G::kPlaneBytes, bar);
    }
    const cx<float>* tw = twiddles<G>(a, tile);
    const Quad q = a.quads[a.t0 + t];
    if (threadIdx.x == 32) prefetch_planes(a, q, (long long)z * NN, (uint32_t)(NN * 4), N3, true);
    __syncthreads();
    // every thread waits (bounded); a time-out anywhere makes the whole block
    // return, after one more bounded wait for the copy in flight
    if (!mbar_wait_bounded(bar, 0, a.err, 1)) *timed_out = 1;
    __syncthreads();
    if (*timed_out) {
        mbar_wait_bounded(bar, 0, nullptr, 0);
        return;
    }
    inv_accum_plane<N, F0, TPL>(a, q, z, tile, tw, reinterpret_cast<double*>(tile),
                       a.e_part != nullptr ? a.e_part + ((long long)(a.t0 + t) * gridDim.x + z) * 2 : nullptr);
}

template <void (*k)(PassArgs), bool max_carveout>
cudaError_t launch_plane(size_t smem, int n, int nt, const PassArgs& a, int batch, cudaStream_t st) {
    if (smem > 48 * 1024) {
        static std::atomic<unsigned long long> done{0};
        cudaError_t e = kernel_limits((const void*)k, (int)smem, max_carveout, done);
        if (e != cudaSuccess) return e;
    }
    dim3 grid((unsigned)n, (unsigned)batch);
    k<<<grid, nt, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace plane_detail

// which: 0 = pair product + forward plane FFT (transposed planes out),
// 1 = inverse plane FFT + accumulation; 2, 3 = the same two passes with natural
// planes, the tile's own layout (the hybrid variant)
template <int N, int F0 = 0>
cudaError_t tplane_launch(int which, const PassArgs& a, int batch, cudaStream_t st) {
    using namespace plane_detail;
    constexpr int TPL = plane_tpl<N>();
    using G = Geo<N, F0, TPL>;
    if (which == 2) return launch_plane<pair_fwd<N, true, F0, TPL>, G::HALF>(G::smem, N, G::NT, a, batch, st);
    if (which == 3) return launch_plane<inv_accum_natural<N, F0, TPL>, G::HALF>(G::smem, N, G::NT, a, batch, st);
    if constexpr (!tplane_supported(N)) {
        return cudaErrorInvalidValue;  // no transposed planes
    } else {
        if (which == 0) return launch_plane<pair_fwd<N, false, F0, TPL>, G::HALF>(G::smem, N, G::NT, a, batch, st);
        return launch_plane<inv_accum<N, F0, TPL>, G::HALF>(G::smem, N, G::NT, a, batch, st);
    }
}

}  // namespace ace
