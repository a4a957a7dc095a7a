// generic.cuh -- the FFT passes of single-precision boxes without compile-time
// kernels: any n0 x n1 x n2 of factors 2, 3, 5 whose x-y plane fits one block's
// shared memory.  The sizes are runtime values; the radix of every stage is
// dispatched to its codelet, and what the compile-time kernels gain from
// constants is gained here from the mapping instead:
//
//   planes   a thread owns a line's butterfly, a warp's lanes run across
//            neighbouring lines (no index divisions inside a butterfly, coalesced
//            rows); the shared plane has an odd row pitch, so lanes along a row
//            and lanes down a column both meet distinct banks.  Forward: product
//            of the functions into the tile, x stages, y stages, the last y stage
//            straight to the spectrum.  Inverse: the first y stage straight from
//            the spectrum, y stages, x stages, then the exchange accumulation
//            (or the split into two real functions) from the tile.
//   pencils  one warp per 128 bytes of every z row (pairs of pencils in packed
//            arithmetic where a z row holds an even count, else single pencils),
//            lanes sharing a pencil's butterflies, no block barriers; forward
//            stages, the Coulomb factors between the last forward and the first
//            inverse stage, inverse stages; or one direction alone.
//
// Bound: instruction issue (runtime strides, about 1.6 times the compile-time
// kernels' instructions per element).  Against the runtime-size tile passes these
// replace, per 32 transforms of 72^3: forward planes 62 vs 127 us, pencils 48 vs
// 347, inverse planes 93 vs 150; 64 orbitals there 6.4 vs 19.8 ms per build, 27
// orbitals on 40 x 48 x 45 0.50 vs 1.31 ms.
#pragma once

#include "internal.h"
#include "pass_kernel.cuh"
#include "tma.cuh"

namespace ace {
namespace generic_detail {

using pass_detail::V4;
using pass_detail::dot4;
using pass_detail::fma4;
using pass_detail::ld4;
using pass_detail::mul4;
using pass_detail::red4;

// Division of small non-negative integers by a runtime constant:
// floor(x / d) for x d < 2^32.
struct FastDiv {
    unsigned m;
    int d;
    __device__ __forceinline__ explicit FastDiv(int dd) : m(dd > 1 ? 0xffffffffu / (unsigned)dd + 1u : 0u), d(dd) {}
    __device__ __forceinline__ int div(int x) const { return d > 1 ? (int)__umulhi((unsigned)x, m) : x; }
};

// f(std::integral_constant<int, r>) for the codelet radix r
template <class F>
__device__ __forceinline__ void with_radix(int r, F&& f) {
    switch (r) {
        case 2: f(std::integral_constant<int, 2>{}); break;
        case 3: f(std::integral_constant<int, 3>{}); break;
        case 4: f(std::integral_constant<int, 4>{}); break;
        case 5: f(std::integral_constant<int, 5>{}); break;
        case 6: f(std::integral_constant<int, 6>{}); break;
        case 8: f(std::integral_constant<int, 8>{}); break;
        case 9: f(std::integral_constant<int, 9>{}); break;
        case 10: f(std::integral_constant<int, 10>{}); break;
        case 12: f(std::integral_constant<int, 12>{}); break;
        case 15: f(std::integral_constant<int, 15>{}); break;
        default: f(std::integral_constant<int, 16>{}); break;
    }
}

// ---------------------------------------------------------------- planes

// One stage (blocks of Lb, radix RAD) of `lines` lines of length n in the
// tile: element e of line l at l ls + e es.
template <int RAD, int SGN>
__device__ __forceinline__ void plane_stage(cx<float>* tile, int lines, int ls, int es, int n, int Lb,
                                            const cx<float>* tw) {
    const int M = Lb / RAD, ts = n / Lb, total = n / RAD * lines;
    const FastDiv dl(lines), dm(M);
    for (int i = threadIdx.x; i < total; i += blockDim.x) {
        const int b = dl.div(i), line = i - b * lines;
        const int beta = dm.div(b), j = b - beta * M;
        butterfly_core<RAD, SGN, float>(tile + line * ls + (beta * Lb + j) * es, M * es, tw, ts * j, j > 0);
    }
    __syncthreads();
}

// Stages [s0, s1) of a line transform in the tile (forward order for SGN < 0,
// backward for SGN > 0).
template <int SGN>
__device__ __forceinline__ void plane_stages(cx<float>* tile, int lines, int ls, int es, const AxisPlan& P,
                                             const cx<float>* tw, int s0, int s1) {
    int Lb = P.n;
    if (SGN < 0) {
        for (int s = 0; s < s0; ++s) Lb /= P.radix[s];
        for (int s = s0; s < s1; ++s) {
            with_radix(P.radix[s], [&](auto r) { plane_stage<decltype(r)::value, SGN>(tile, lines, ls, es, P.n, Lb, tw); });
            Lb /= P.radix[s];
        }
    } else {
        for (int s = 0; s < s1; ++s) Lb /= P.radix[s];  // length below the last of the stages
        for (int s = s1 - 1; s >= s0; --s) {
            Lb *= P.radix[s];
            with_radix(P.radix[s], [&](auto r) { plane_stage<decltype(r)::value, SGN>(tile, lines, ls, es, P.n, Lb, tw); });
        }
    }
}

constexpr int kPlaneThreads = 768;  // at most (80 registers per thread)

__device__ __forceinline__ void load_twiddles(const PassArgs& a, cx<float>* twx, cx<float>* twy) {
    for (int j = threadIdx.x; j < a.n2; j += blockDim.x) twx[j] = reinterpret_cast<const cx<float>*>(a.twx)[j];
    for (int j = threadIdx.x; j < a.n1; j += blockDim.x) twy[j] = reinterpret_cast<const cx<float>*>(a.twy)[j];
}

// Plane z of transform t: PRO_PAIR (products of four functions) or PRO_PACK2
// (two functions), x and y forward, to the spectrum.
template <int PRO>
__global__ void __launch_bounds__(kPlaneThreads, 1) plane_forward(PassArgs a) {
    extern __shared__ __align__(16) unsigned char smem_gen[];
    const int n1 = a.n1, n2 = a.n2, P = n2 | 1, NN = n1 * n2;
    cx<float>* tile = reinterpret_cast<cx<float>*>(smem_gen);
    cx<float>* twx = tile + n1 * P;
    cx<float>* twy = twx + n2;
    const int z = blockIdx.x, t = blockIdx.y;
    const Quad q = a.quads[a.t0 + t];
    const long long N = (long long)a.n0 * NN, plane0 = (long long)z * NN;
    load_twiddles(a, twx, twy);
    {
        const bool has2 = q.c >= 0;
        const float* fa = reinterpret_cast<const float*>(a.fl) + q.a * N + plane0;
        const float* fb = reinterpret_cast<const float*>(a.fr) + q.b * N + plane0;
        const float* fc = reinterpret_cast<const float*>(a.fl) + (has2 ? q.c : q.a) * N + plane0;
        const float* fd = reinterpret_cast<const float*>(a.fr) + (has2 ? q.d : q.b) * N + plane0;
        if (NN % 4 == 0) {
            // float4 loads along the plane, whole lines; four steps' in flight
            const FastDiv dx(n2);
            const int pad = P - n2;
            constexpr int W = 4;
            for (int k0 = threadIdx.x; k0 < NN / 4; k0 += W * blockDim.x) {
                V4<float> re[W], im[W];
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const int r = 4 * (k0 + w * blockDim.x);
                    im[w] = V4<float>{0.f, 0.f, 0.f, 0.f};
                    if (r < NN) {
                        re[w] = ld4(fa + r);
                        if (PRO == PRO_PAIR) re[w] = mul4(re[w], ld4(fb + r));
                        if (has2) {
                            im[w] = ld4(fc + r);
                            if (PRO == PRO_PAIR) im[w] = mul4(im[w], ld4(fd + r));
                        }
                    }
                }
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    const int r = 4 * (k0 + w * blockDim.x);
                    if (r >= NN) continue;
                    const cx<float> v[4] = {mk(re[w].x, im[w].x), mk(re[w].y, im[w].y), mk(re[w].z, im[w].z),
                                            mk(re[w].w, im[w].w)};
                    tile_write4(tile, r + dx.div(r) * pad, r + 2 + dx.div(r + 2) * pad, v);
                }
            }
        } else {
            const FastDiv dx(n2);
#pragma unroll 8
            for (int i = threadIdx.x; i < NN; i += blockDim.x) {
                float re = __ldg(fa + i), im = has2 ? __ldg(fc + i) : 0.f;
                if (PRO == PRO_PAIR) {
                    re *= __ldg(fb + i);
                    if (has2) im *= __ldg(fd + i);
                }
                tile[i + dx.div(i) * (P - n2)] = mk(re, im);
            }
        }
    }
    __syncthreads();
    plane_stages<-1>(tile, n1, P, 1, a.px, twx, 0, a.px.nstages);
    const int S = a.py.nstages;
    plane_stages<-1>(tile, n2, 1, P, a.py, twy, 0, S - 1);
    // last y stage (adjacent positions, no twiddles): lanes along x write rows
    cx<float>* out = reinterpret_cast<cx<float>*>(a.dst) + t * a.dst_tstride + plane0;
    with_radix(a.py.radix[S - 1], [&](auto rc) {
        constexpr int RAD = decltype(rc)::value;
        const FastDiv dx(n2);
        for (int i = threadIdx.x; i < NN / RAD; i += blockDim.x) {
            const int b = dx.div(i), x = i - b * n2;
            const cx<float>* col = tile + b * RAD * P + x;
            cx<float> u[RAD];
#pragma unroll
            for (int k = 0; k < RAD; ++k) u[k] = col[k * P];
            Dft<RAD, -1, float>::run(u);
            cx<float>* o = out + b * RAD * n2 + x;
#pragma unroll
            for (int k = 0; k < RAD; ++k) o[k * n2] = u[k];
        }
    });
}

// Plane z of transform t: spectrum, y and x inverse, then EPI_ACCUM (exchange
// accumulation and pair energies) or EPI_SPLIT (two real functions, scaled).
template <int EPI>
__global__ void __launch_bounds__(kPlaneThreads, 1) plane_inverse(PassArgs a) {
    extern __shared__ __align__(16) unsigned char smem_gen[];
    __shared__ double red[2 * (kPlaneThreads / 32)];
    const int n1 = a.n1, n2 = a.n2, P = n2 | 1, NN = n1 * n2;
    cx<float>* tile = reinterpret_cast<cx<float>*>(smem_gen);
    cx<float>* twx = tile + n1 * P;
    cx<float>* twy = twx + n2;
    const int z = blockIdx.x, t = blockIdx.y;
    const Quad q = a.quads[a.t0 + t];
    const long long N = (long long)a.n0 * NN, plane0 = (long long)z * NN;
    load_twiddles(a, twx, twy);
    const int S = a.py.nstages;
    const cx<float>* in = reinterpret_cast<const cx<float>*>(a.src) + t * a.src_tstride + plane0;
    with_radix(a.py.radix[S - 1], [&](auto rc) {
        constexpr int RAD = decltype(rc)::value;
        const FastDiv dx(n2);
        for (int i = threadIdx.x; i < NN / RAD; i += blockDim.x) {
            const int b = dx.div(i), x = i - b * n2;
            const cx<float>* o = in + b * RAD * n2 + x;
            cx<float> u[RAD];
#pragma unroll
            for (int k = 0; k < RAD; ++k) {
                const float2 v = __ldg(reinterpret_cast<const float2*>(o + k * n2));
                u[k] = mk(v.x, v.y);
            }
            Dft<RAD, +1, float>::run(u);
            cx<float>* col = tile + b * RAD * P + x;
#pragma unroll
            for (int k = 0; k < RAD; ++k) col[k * P] = u[k];
        }
    });
    __syncthreads();
    plane_stages<+1>(tile, n2, 1, P, a.py, twy, 0, S - 1);
    plane_stages<+1>(tile, n1, P, 1, a.px, twx, 0, a.px.nstages);

    const bool has2 = q.c >= 0;
    float* wa_p = reinterpret_cast<float*>(a.accl) + q.a * N + plane0;
    float* wc_p = reinterpret_cast<float*>(a.accl) + (has2 ? q.c : q.a) * N + plane0;
    if (EPI == EPI_SPLIT) {
        const float s = (float)a.scale;
        const FastDiv dx(n2);
#pragma unroll 4
        for (int i = threadIdx.x; i < NN; i += blockDim.x) {
            const cx<float> v = tile[i + dx.div(i) * (P - n2)];
            wa_p[i] = v.re * s;
            if (has2) wc_p[i] = v.im * s;
        }
        return;
    }
    const bool share = has2 && q.c == q.a, sym = a.symmetric != 0;
    const bool upd_b = sym && q.a != q.b, upd_d = sym && has2 && q.c != q.d;
    const float* la_p = reinterpret_cast<const float*>(a.fl) + q.a * N + plane0;
    const float* rb_p = reinterpret_cast<const float*>(a.fr) + q.b * N + plane0;
    const float* lc_p = reinterpret_cast<const float*>(a.fl) + (has2 ? q.c : q.a) * N + plane0;
    const float* rd_p = reinterpret_cast<const float*>(a.fr) + (has2 ? q.d : q.b) * N + plane0;
    float* wb_p = sym ? reinterpret_cast<float*>(a.accr) + q.b * N + plane0 : nullptr;
    float* wd_p = sym ? reinterpret_cast<float*>(a.accr) + (has2 ? q.d : q.b) * N + plane0 : nullptr;
    float e1 = 0.f, e2 = 0.f;
    if (NN % 4 == 0) {
        // four values per step along the plane, every load and reduction in
        // whole lines; the loads of two steps are issued before their updates
        // (ordered operations)
        const FastDiv dx(n2);
        const int pad = P - n2;
        constexpr int W = 2;
        for (int k0 = threadIdx.x; k0 < NN / 4; k0 += W * blockDim.x) {
            V4<float> la[W], rb[W], lc[W], rd[W];
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const int r = 4 * (k0 + w * blockDim.x);
                if (r < NN) {
                    la[w] = ld4(la_p + r);
                    rb[w] = ld4(rb_p + r);
                    if (has2) {
                        lc[w] = share ? la[w] : ld4(lc_p + r);
                        rd[w] = ld4(rd_p + r);
                    }
                }
            }
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const int r = 4 * (k0 + w * blockDim.x);
                if (r >= NN) continue;
                cx<float> v[4];
                tile_read4(tile, r + dx.div(r) * pad, r + 2 + dx.div(r + 2) * pad, v);
                const V4<float> v1 = {v[0].re, v[1].re, v[2].re, v[3].re}, v2 = {v[0].im, v[1].im, v[2].im, v[3].im};
                V4<float> wa = mul4(v1, rb[w]);
                e1 += dot4(mul4(la[w], rb[w]), v1);
                if (has2) {
                    e2 += dot4(mul4(lc[w], rd[w]), v2);
                    if (share)
                        wa = fma4(v2, rd[w], wa);
                    else
                        red4(wc_p + r, mul4(v2, rd[w]));
                    if (upd_d) red4(wd_p + r, mul4(v2, lc[w]));
                }
                red4(wa_p + r, wa);
                if (upd_b) red4(wb_p + r, mul4(v1, la[w]));
            }
        }
    } else {
        const FastDiv dx(n2);
        for (int i = threadIdx.x; i < NN; i += blockDim.x) {
            const float la = __ldg(la_p + i), rb = __ldg(rb_p + i);
            const cx<float> v = tile[i + dx.div(i) * (P - n2)];
            float wa = v.re * rb;
            e1 += la * rb * v.re;
            if (has2) {
                const float lc = share ? la : __ldg(lc_p + i), rd = __ldg(rd_p + i);
                e2 += lc * rd * v.im;
                if (share)
                    wa += v.im * rd;
                else
                    atomicAdd(wc_p + i, v.im * rd);
                if (upd_d) atomicAdd(wd_p + i, v.im * lc);
            }
            atomicAdd(wa_p + i, wa);
            if (upd_b) atomicAdd(wb_p + i, v.re * la);
        }
    }
    if (a.e_part != nullptr) {
        const double d1 = warp_sum_ff(e1), d2 = warp_sum_ff(e2);
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
        if (lane == 0) {
            red[2 * warp] = d1;
            red[2 * warp + 1] = d2;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double s1 = 0, s2 = 0;
            for (int w = 0; w < nw; ++w) {
                s1 += red[2 * w];
                s2 += red[2 * w + 1];
            }
            double* dst = a.e_part + ((long long)(a.t0 + t) * gridDim.x + z) * 2;
            dst[0] = s1;
            dst[1] = s2;
        }
    }
}

// ---------------------------------------------------------------- pencils
// V = f2: units of two neighbouring pencils (16 bytes), 8 per warp; V = float:
// single pencils (8 bytes), 16 per warp.  col: this lane's unit in the shared
// [n0][U] buffer; lane h of the L that share it takes butterflies h, h + L, ...

template <typename V>
struct Units {
    static constexpr int U = sizeof(V) == 8 ? 8 : 16, L = 32 / U;
};

__device__ __forceinline__ void async_unit(void* smem_dst, const cx<f2>* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(smem_dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void async_unit(void* smem_dst, const cx<float>* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(smem_dst)), "l"(src) : "memory");
}
// two neighbouring complex values <-> their real and imaginary parts paired
__device__ __forceinline__ cx<f2> turn_unit(cx<f2> a) {
    return mk(mk_f2(lo(a.re), lo(a.im)), mk_f2(hi(a.re), hi(a.im)));
}
__device__ __forceinline__ cx<float> turn_unit(cx<float> a) { return a; }
__device__ __forceinline__ void load_factor(const float* p, f2& k) {
    k.v = __ldg(reinterpret_cast<const unsigned long long*>(p));
}
__device__ __forceinline__ void load_factor(const float* p, float& k) { k = __ldg(p); }

template <int RAD, int SGN, typename V>
__device__ __forceinline__ void pencil_stage(cx<V>* col, int n, int Lb, const cx<float>* tw, int h) {
    constexpr int U = Units<V>::U, L = Units<V>::L;
    const int M = Lb / RAD, ts = n / Lb;
    const FastDiv dm(M);
#pragma unroll 1
    for (int i = h; i < n / RAD; i += L) {
        const int beta = dm.div(i), j = i - beta * M;
        cx<V>* base = col + (beta * Lb + j) * U;
        cx<V> u[RAD];
#pragma unroll
        for (int q = 0; q < RAD; ++q) u[q] = base[q * M * U];
        if (SGN > 0 && j > 0) {
#pragma unroll
            for (int q = 1; q < RAD; ++q) {
                cx<float> w = tw[q * ts * j];
                w.im = -w.im;
                u[q] = cmul(u[q], w);
            }
        }
        Dft<RAD, SGN, V>::run(u);
        if (SGN < 0 && j > 0) {
#pragma unroll
            for (int q = 1; q < RAD; ++q) u[q] = cmul(u[q], tw[q * ts * j]);
        }
#pragma unroll
        for (int q = 0; q < RAD; ++q) base[q * M * U] = u[q];
    }
    __syncwarp();
}

// MODE: -1 forward z, +1 inverse z, 0 forward, Coulomb factors, inverse.
template <typename V, int MODE>
__global__ void __launch_bounds__(32) pencils(PassArgs a, int units) {
    constexpr int U = Units<V>::U, L = Units<V>::L;
    extern __shared__ __align__(16) unsigned char smem_gen[];
    cx<V>* buf = reinterpret_cast<cx<V>*>(smem_gen);
    cx<float>* tw = reinterpret_cast<cx<float>*>(buf + a.n0 * U);
    const int lane = threadIdx.x, l = lane % U, h = lane / U, n = a.n0;
    const int p = blockIdx.x * U + l;
    const bool on = p < units;  // lanes past the last unit only keep the barriers
    const int t = blockIdx.y;
    const cx<V>* src = reinterpret_cast<const cx<V>*>(reinterpret_cast<const cx<float>*>(a.src) + t * a.src_tstride) + p;
    cx<V>* dst = reinterpret_cast<cx<V>*>(reinterpret_cast<cx<float>*>(a.dst) + t * a.dst_tstride) + p;
    if (on)
#pragma unroll 4
        for (int z = h; z < n; z += L) async_unit(buf + z * U + l, src + (long long)z * units);
    for (int j = lane; j < n; j += 32) tw[j] = reinterpret_cast<const cx<float>*>(a.twz)[j];
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    cx<V>* col = buf + l;
    if (sizeof(V) == 8) {  // {re0, im0, re1, im1} -> {re0, re1, im0, im1}
        if (on)
            for (int z = h; z < n; z += L) col[z * U] = turn_unit(col[z * U]);
        __syncwarp();
    }
    const int hh = on ? h : n;  // no butterflies past the last unit
    const AxisPlan& P = a.pz;
    int Lb = n;
    if (MODE <= 0) {
        const int last = MODE == 0 ? P.nstages - 1 : P.nstages;
        for (int s = 0; s < last; ++s) {
            with_radix(P.radix[s], [&](auto r) { pencil_stage<decltype(r)::value, -1, V>(col, n, Lb, tw, hh); });
            Lb /= P.radix[s];
        }
    }
    if (MODE == 0) {
        with_radix(P.radix[P.nstages - 1], [&](auto r) {
            constexpr int RAD = decltype(r)::value;
            const float* kern = reinterpret_cast<const float*>(a.kern) + (sizeof(V) / 4) * p;
            const long long ks = (long long)units * (sizeof(V) / 4);
#pragma unroll 1
            for (int b = hh; b < n / RAD; b += L) {
                V k[RAD];
                cx<V> u[RAD];
#pragma unroll
                for (int q = 0; q < RAD; ++q) load_factor(kern + (b * RAD + q) * ks, k[q]);
#pragma unroll
                for (int q = 0; q < RAD; ++q) u[q] = col[(b * RAD + q) * U];
                Dft<RAD, -1, V>::run(u);
#pragma unroll
                for (int q = 0; q < RAD; ++q) u[q] = scale(u[q], k[q]);
                Dft<RAD, +1, V>::run(u);
#pragma unroll
                for (int q = 0; q < RAD; ++q) col[(b * RAD + q) * U] = u[q];
            }
        });
        __syncwarp();
    }
    if (MODE >= 0) {
        Lb = MODE == 0 ? P.radix[P.nstages - 1] : 1;
        for (int s = MODE == 0 ? P.nstages - 2 : P.nstages - 1; s >= 0; --s) {
            Lb *= P.radix[s];
            with_radix(P.radix[s], [&](auto r) { pencil_stage<decltype(r)::value, +1, V>(col, n, Lb, tw, hh); });
        }
    }
    if (on)
#pragma unroll 4
        for (int z = h; z < n; z += L) dst[(long long)z * units] = turn_unit(col[z * U]);
}

// ------------------------------------------------- pencils of the sphere
// The z transforms of the orbitals and of W touch the cutoff sphere only: of the
// plane's pencils about a quarter hold plane waves.  off[p] .. off[p + 1] are
// the entries of pencil p, each {z position, plane wave i for +G or ~i for -G}.

// Orbitals to half-real space: the coefficients of a quad's two orbitals
// (Z(G) = c_a + i c_b, Z(-G) = c_a^* + i c_b^*) gathered into shared columns,
// inverse z, to the box; groups without plane waves only write zeros.  Replaces
// a cleared box, a scatter and a z pass over it (334 us per 64 transforms of
// 96^3); bound by the box's writes.
template <typename V>
__global__ void __launch_bounds__(32) sphere_inverse(PassArgs a, int units, SphereArgs sp) {
    constexpr int U = Units<V>::U, L = Units<V>::L, W = sizeof(V) / 4;
    extern __shared__ __align__(16) unsigned char smem_gen[];
    cx<V>* buf = reinterpret_cast<cx<V>*>(smem_gen);
    cx<float>* tw = reinterpret_cast<cx<float>*>(buf + a.n0 * U);
    const int lane = threadIdx.x, l = lane % U, h = lane / U, n = a.n0;
    const int p = blockIdx.x * U + l, t = blockIdx.y;
    const bool on = p < units;
    cx<V>* dst = reinterpret_cast<cx<V>*>(reinterpret_cast<cx<float>*>(a.dst) + t * a.dst_tstride) + p;
    const int e0 = on ? sp.off[p * W] : 0, e2 = on ? sp.off[p * W + W] : 0, e1 = on ? sp.off[p * W + 1] : 0;
    cx<V> zero;
    zero.re = zero.im = V(0.0);
    if (!__any_sync(0xffffffffu, e2 > e0)) {
        if (on)
            for (int z = h; z < n; z += L) dst[(long long)z * units] = zero;
        return;
    }
    const Quad q = a.quads[a.t0 + t];
    for (int j = lane; j < n; j += 32) tw[j] = reinterpret_cast<const cx<float>*>(a.twz)[j];
    for (int z = h; z < n; z += L) buf[z * U + l] = zero;
    __syncwarp();
    const cx<float>* pa = reinterpret_cast<const cx<float>*>(sp.psi) + (long long)q.a * sp.npw;
    const cx<float>* pb = reinterpret_cast<const cx<float>*>(sp.psi) + (long long)(q.c >= 0 ? q.c : q.a) * sp.npw;
    for (int e = e0 + h; e < e2; e += L) {
        const int2 en = sp.ent[e];
        const bool neg = en.y < 0;
        const int i = neg ? ~en.y : en.y;
        const cx<float> ca = pa[i], cb = q.c >= 0 ? pb[i] : mk(0.f, 0.f);
        const cx<float> v = neg ? mk(ca.re + cb.im, cb.re - ca.im) : mk(ca.re - cb.im, ca.im + cb.re);
        float* u = reinterpret_cast<float*>(buf + en.x * U + l);
        const int w = e >= e1 ? W - 1 : 0;
        u[w] = v.re;
        u[W + w] = v.im;
    }
    __syncwarp();
    const AxisPlan& P = a.pz;
    const int hh = e2 > e0 ? h : n;  // columns without plane waves stay zero
    int Lb = 1;
    for (int s = P.nstages - 1; s >= 0; --s) {
        Lb *= P.radix[s];
        with_radix(P.radix[s], [&](auto r) { pencil_stage<decltype(r)::value, +1, V>(buf + l, n, Lb, tw, hh); });
    }
    if (on)
#pragma unroll 4
        for (int z = h; z < n; z += L) dst[(long long)z * units] = turn_unit(buf[z * U + l]);
}

// The forward z transform of the pencils (units sp.list[0 .. nlist)) that hold
// plane waves; only those entries of the box are written (in place).
template <typename V>
__global__ void __launch_bounds__(32) sphere_forward(PassArgs a, int units, SphereArgs sp) {
    constexpr int U = Units<V>::U, L = Units<V>::L, W = sizeof(V) / 4;
    extern __shared__ __align__(16) unsigned char smem_gen[];
    cx<V>* buf = reinterpret_cast<cx<V>*>(smem_gen);
    cx<float>* tw = reinterpret_cast<cx<float>*>(buf + a.n0 * U);
    const int lane = threadIdx.x, l = lane % U, h = lane / U, n = a.n0;
    const int g = blockIdx.x * U + l, t = blockIdx.y;
    const bool on = g < sp.nlist;
    const int p = on ? sp.list[g] : 0;
    cx<float>* box = reinterpret_cast<cx<float>*>(a.dst) + t * a.dst_tstride;
    const cx<V>* src = reinterpret_cast<const cx<V>*>(reinterpret_cast<const cx<float>*>(a.src) + t * a.src_tstride) + p;
    if (on)
#pragma unroll 4
        for (int z = h; z < n; z += L) async_unit(buf + z * U + l, src + (long long)z * units);
    for (int j = lane; j < n; j += 32) tw[j] = reinterpret_cast<const cx<float>*>(a.twz)[j];
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    if (W == 2) {
        if (on)
            for (int z = h; z < n; z += L) buf[z * U + l] = turn_unit(buf[z * U + l]);
        __syncwarp();
    }
    const AxisPlan& P = a.pz;
    const int hh = on ? h : n;
    int Lb = n;
    for (int s = 0; s < P.nstages; ++s) {
        with_radix(P.radix[s], [&](auto r) { pencil_stage<decltype(r)::value, -1, V>(buf + l, n, Lb, tw, hh); });
        Lb /= P.radix[s];
    }
    if (!on) return;
    const int e0 = sp.off[p * W], e1 = sp.off[p * W + 1], e2 = sp.off[p * W + W];
    for (int e = e0 + h; e < e2; e += L) {
        const int z = sp.ent[e].x, w = e >= e1 ? W - 1 : 0;
        const float* u = reinterpret_cast<const float*>(buf + z * U + l);
        box[(long long)z * units * W + p * W + w] = mk(u[w], u[W + w]);
    }
}

}  // namespace generic_detail
}  // namespace ace
