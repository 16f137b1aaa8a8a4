// conv_wide.cuh -- the separable convolution on large tiles, 56 x 120 outputs, for
// one application of H to a large image.
//
// GB300, 2160 x 3840, r = 6: 32.8 -> 26.3 us; 4096^2, r = 10: 70 -> 60 us (66 MB and
// 134 MB would take 10 and 20 us; issue slots are two thirds busy).  The level
// solvers keep the 32 x 64 tiles: with these, a 4096^2 solve was as fast (367 us
// against 367 at r = 10, 340 against 325 at r = 6), a 2048^2 one slower (149 against
// 136: 666 tiles leave the third round of 304 blocks mostly idle).
// A 32 x 64 tile (conv_tile.cuh) computes its vertical pass on 1.3 times its columns
// at r = 10, reads 31 staged values for 11 outputs of a column and stages its
// result in shared memory once more to store it by rows: 78 instructions a pixel,
// four barriers per 2048 pixels.  Here a thread of the vertical pass owns four
// columns of 8 rows (28 16-byte loads for 32 outputs; 36 quads x 7 groups keep 252
// of 256 threads busy at the largest radius), the horizontal pass owns four
// columns of a row and stores them itself: two barriers per 6720 pixels.  A block
// takes one tile; the other blocks of its SM run while its window arrives by cp.async.
// Each output sums its taps in increasing order, vertical pass first, as in
// conv_tile.cuh (the same value).
#pragma once

#include "launch.hpp"

namespace eecmg {

template <int R>
struct Wide {
    static constexpr int WH = 56, WW = 120, VR = 8, GR = WH / VR;
    static constexpr int PADX = (R + 3) / 4 * 4, AX = WW + 2 * PADX, QX = AX / 4, NY = WH + 2 * R;
    static constexpr int IN = NY * AX, TMP = WH * AX, NT = 2 * R + 1;
    static constexpr size_t bytes = sizeof(float) * (size_t)(IN + TMP);
    static_assert(QX * GR <= NTHREADS, "one round of the vertical pass");
};
constexpr int WIDE_H = Wide<0>::WH, WIDE_W = Wide<0>::WW;

// Copies the window of the tile at (y0, x0) into A (zero outside the image): 16-byte
// asynchronous copies through L2, or single loads where x is not 16-byte aligned.
template <int R>
__device__ __forceinline__ void wide_stage(const float* __restrict__ x, int h, int w, int y0, int x0, float* A, bool vec) {
    using W = Wide<R>;
    const unsigned int base = (unsigned int)__cvta_generic_to_shared(A);
    for (int c = threadIdx.x; c < W::NY * W::QX; c += NTHREADS) {
        const int r = c / W::QX, q = c - r * W::QX;
        const int gy = y0 - R + r, gx = x0 - W::PADX + 4 * q;
        const bool in = gy >= 0 && gy < h && gx >= 0 && gx < w;
        const float* g = in ? x + (size_t)gy * w + gx : x;
        if (vec) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(base + 16u * (unsigned int)c), "l"(g),
                         "r"(in ? 16 : 0)
                         : "memory");
        } else {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (in) v = make_float4(__ldcg(g), __ldcg(g + 1), __ldcg(g + 2), __ldcg(g + 3));
            reinterpret_cast<float4*>(A)[c] = v;
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// tmp(r, c) = sum_d cy[d] A(r + d, c) over the window's columns.
template <int R>
__device__ __forceinline__ void wide_vertical(const float* A, float* tmp, const float* cy) {
    using W = Wide<R>;
    const int q = threadIdx.x % W::QX, g = threadIdx.x / W::QX;
    if (g >= W::GR) return;
    const float4* a = reinterpret_cast<const float4*>(A) + g * W::VR * W::QX + q;
    float4 acc[W::VR];
#pragma unroll
    for (int i = 0; i < W::VR; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int j = 0; j < W::VR + 2 * R; ++j) {
        const float4 v = a[j * W::QX];
#pragma unroll
        for (int i = 0; i < W::VR; ++i)
            if (j - i >= 0 && j - i <= 2 * R) acc[i] = fma4(cy[j - i], v, acc[i]);
    }
    float4* t = reinterpret_cast<float4*>(tmp) + g * W::VR * W::QX + q;
#pragma unroll
    for (int i = 0; i < W::VR; ++i) t[i * W::QX] = acc[i];
}

// The convolution of tile t: epi(index, (C (*) x) of four pixels); w a multiple of 4.
// sm: Wide<R>::bytes; cy, cx: the taps centred at R in shared memory.  Called by all
// threads of the block.
template <int R, class Epi>
__device__ __forceinline__ void wide_conv(float* sm, const float* cy, const float* cx, const float* x, int h, int w,
                                          int t, Epi&& epi) {
    using W = Wide<R>;
    float* A = sm;
    float* tmp = sm + W::IN;
    const int tx = (w + W::WW - 1) / W::WW, y0 = (t / tx) * W::WH, x0 = (t % tx) * W::WW;
    wide_stage<R>(x, h, w, y0, x0, A, (reinterpret_cast<uintptr_t>(x) & 15) == 0);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // the window and the taps
    wide_vertical<R>(A, tmp, cy);
    __syncthreads();
    float c[W::NT];
#pragma unroll
    for (int d = 0; d < W::NT; ++d) c[d] = cx[d];
#pragma unroll 1
    for (int i = threadIdx.x; i < W::WH * (W::WW / 4); i += NTHREADS) {
        const int r = i / (W::WW / 4), q = i - r * (W::WW / 4);
        const int gy = y0 + r, gx = x0 + 4 * q;
        if (gy >= h || gx >= w) continue;
        constexpr int NQ = 1 + 2 * W::PADX / 4;
        const float4* s = reinterpret_cast<const float4*>(tmp) + r * W::QX + q;
        float v[4 * NQ];
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            const float4 u = s[j];
            v[4 * j] = u.x;
            v[4 * j + 1] = u.y;
            v[4 * j + 2] = u.z;
            v[4 * j + 3] = u.w;
        }
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int d = 0; d < W::NT; ++d) {
            constexpr int b = W::PADX - R;
            o.x = fmaf(c[d], v[b + d], o.x);
            o.y = fmaf(c[d], v[b + d + 1], o.y);
            o.z = fmaf(c[d], v[b + d + 2], o.z);
            o.w = fmaf(c[d], v[b + d + 3], o.w);
        }
        epi((size_t)gy * w + gx, o);
    }
}

}  // namespace eecmg
