// volume_impl.cuh -- the level solve of the volume path (internal): the
// convolution tile and the persistent MR-II kernel, templated on the level
// PSF's radius R.  The instantiations R = 0 .. EECMG_VOL_MAX_RADIUS are split
// over the volume_r*.cu translation units (compile time); volume.cu holds the
// voxel kernels of the level start, the planner and the C ABI.
#pragma once

#include <cstdint>

#include "../../include/eecmg.h"
#include "common.cuh"
#include "persistent.cuh"

namespace eecmg {
namespace vol {

constexpr int VR = EECMG_VOL_MAX_RADIUS;
constexpr int VK = 2 * VR + 1;
constexpr int MX = 64;                  // columns of a marched tile
constexpr int TX = 32, TY = 8, TZ = 8;  // small and sparse forms: output tile (columns, rows, slices)

// How a level's PSF is applied (fixed by the planner from its taps).
enum VolForm : int {
    VF_SEP = 0,     // an outer product of three factors: three 1-D passes
    VF_DENSE = 1,   // rows of 2 r + 1 taps for every (slice, row) offset that has one
    VF_SPARSE = 2,  // a list of taps
    VF_SMALL = 3,   // as VF_SEP, on a level with few slices per block to march
};

// Taps of one level in correlation form, y(v) = sum_d C(d) x(v + d), C(d) = K(-d),
// centred at r = the level PSF's largest radius (shorter axes padded with zeros).
struct VolTaps {
    int r;
    int form;                      // VolForm
    float cz[VK], cy[VK], cx[VK];  // VF_SEP, VF_SMALL: factors, index d + r
    int ntap;                      // else: taps in the job's tap list
};

struct VolJob {
    int d, h, w;
    long long n;    // voxels
    long long n4;   // padded voxels / 4
    const float* g;
    float* u;
    float* R;
    float* P[3];
    float* Q[3];
    float* Z;
    VolTaps taps;
    const int4* gtaps;  // VF_DENSE, VF_SPARSE: (dz, dy, dx, weight bits)
    int m;
    int zero_start;
    double stop_tol;    // discrepancy: stop once ||r||_RMS <= stop_tol (0: off)
    double conv_tol;    // stop once ||r|| <= conv_tol ||g|| (0: off)
    double* partials;
    GroupSync* gs;
    double* out;        // [0] iterations, [1] ||r||^2, [2] stop reason
};

// Per-block replica of the solve's scalars (identical in every block), in FP64.  A
// dependent FP64 operation takes 66 cycles on GB300, so a phase takes at most one
// quotient (its two are independent) and no root: the stop test is on ||r||^2.
struct VolScal {
    double rr, qq, qqp, qqn, lim2;
    float a, b1, b2;
    int k, done;
};

// per-thread compensated sum (cascaded: the rounding errors are kept in lo)
__device__ __forceinline__ void acc_add(DF& a, float v) {
    const DF s = two_sum(a.hi, v);
    a.hi = s.hi;
    a.lo += s.lo;
}

// ------------------------------------------------------------- convolution
//
// A convolution phase divides the level's slices of MX x MY column tiles evenly
// over the blocks: block b takes a contiguous range of the (tile, slice) pairs,
// and within a tile marches along the slices.  A ring of input planes (the tile
// with an r-voxel halo, zero outside the volume) is filled by cp.async three
// slices ahead; one barrier per slice.
// VF_SEP: a thread owns four columns of one or two rows, halo columns included.
// The rows pass reads the staged plane; its result enters the 2 r + 1 outputs along
// the slices it contributes to, kept as partial sums in registers; a finished
// slice goes through shared memory once for the columns pass, one slice behind.
// So a voxel costs 3 (2 r + 1) multiplications, about a quarter of a shared
// load per multiplication and no index arithmetic beyond its row.
// VF_DENSE: the thread's window of each row enters all 2 r + 1 slices' partial sums.
// A range repeats the 2 r slices around its start: at 256^3 and r = 3, 6 to 34 (VF_SEP,
// 10 x 4 tiles of 28 rows) or to 54 (VF_DENSE, 16 x 4 of 16 rows) of its own.
// What a phase does with H x: out = H x (or a - H x) and its sums.
enum VolEpi : int { VE_RESID = 0, VE_STORE, VE_Q1, VE_Z };
struct EpiArgs {
    const float* a;  // VE_RESID: g; VE_Q1: r; VE_Z: q_k
    const float* b;  // VE_Z: q_{k-1} (NULL: none)
    float* out;
    int mode;
};

__device__ __forceinline__ float4 ld_quad(const float* p, size_t i, int nv, bool vec) {
    if (vec) return __ldcg(reinterpret_cast<const float4*>(p + i));
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    r.x = __ldcg(p + i);
    if (nv > 1) r.y = __ldcg(p + i + 1);
    if (nv > 2) r.z = __ldcg(p + i + 2);
    if (nv > 3) r.w = __ldcg(p + i + 3);
    return r;
}

// The products of four pairs into a compensated sum, one at a time: a sum of them in
// plain FP32 would lose what the compensation keeps.
__device__ __forceinline__ void acc_dot(DF& s, float4 a, float4 b) {
    acc_add(s, a.x * b.x);
    acc_add(s, a.y * b.y);
    acc_add(s, a.z * b.z);
    acc_add(s, a.w * b.w);
}
__device__ __forceinline__ void acc_dot(DF& s, float a, float b) { acc_add(s, a * b); }
__device__ __forceinline__ float sub(float a, float b) { return a - b; }
__device__ __forceinline__ float4 sub(float4 a, float4 b) {
    return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}

// What a phase stores for one (T = float) or four outputs of a row, and their products
// into the phase's sums.
template <class T>
__device__ __forceinline__ T epilogue(const EpiArgs& E, T hx, T a, T b, DF (&acc)[2]) {
    if (E.mode == VE_RESID) {
        const T o = sub(a, hx);
        acc_dot(acc[0], o, o);
        acc_dot(acc[1], a, a);
        return o;
    }
    if (E.mode == VE_Q1) {
        acc_dot(acc[0], hx, hx);
        acc_dot(acc[1], a, hx);
    } else if (E.mode == VE_Z) {
        acc_dot(acc[0], a, hx);
        acc_dot(acc[1], b, hx);
    }
    return hx;
}
// Four outputs of a row at element i, of which nv (1..4) lie in the volume.
__device__ __forceinline__ void epilogue4(const EpiArgs& E, size_t i, int nv, bool vec, float4 hx, float4 a,
                                          float4 b, DF (&acc)[2]) {
    if (nv < 4) hx.w = a.w = 0.f;
    if (nv < 3) hx.z = a.z = 0.f;
    if (nv < 2) hx.y = a.y = 0.f;
    const float4 o = epilogue(E, hx, a, b, acc);
    if (vec) {
        *reinterpret_cast<float4*>(E.out + i) = o;
    } else {
        E.out[i] = o.x;
        if (nv > 1) E.out[i + 1] = o.y;
        if (nv > 2) E.out[i + 2] = o.z;
        if (nv > 3) E.out[i + 3] = o.w;
    }
}

template <int R>
struct March {
    // a staged row starts PADX = R rounded up to 4 voxels left of the tile, so
    // rows are whole 16-byte chunks
    static constexpr int PADX = (R + 3) / 4 * 4;
    static constexpr int AX = MX + 2 * PADX, QX = AX / 4;  // a staged row, in floats and in quads
    static constexpr int RING = 4;
    // VF_SEP: RPT rows per thread (two quads of 2 r partial sums fit the registers up to
    // r = 4), QX quads x GR row groups of threads
    static constexpr int RPT = R <= 4 ? 2 : 1, GR = NTHREADS / QX, SY = GR * RPT;
    static constexpr int SPLANE = (SY + 2 * R) * AX, V = SY * AX;
    // VF_DENSE: 16 quads x 16 rows of threads
    static constexpr int DY = NTHREADS / (MX / 4), DPLANE = (DY + 2 * R) * AX;
    static constexpr int NW4 = (2 * R + 1 + 3) / 4;        // a row of taps, padded to float4
    static constexpr int WTS = (2 * R + 1) * (2 * R + 1) * NW4 * 4;
    static constexpr size_t bytes(int form) {
        return sizeof(float) * (form == VF_SEP ? RING * (size_t)SPLANE + 2 * V : RING * (size_t)DPLANE + WTS + 16);
    }
    static constexpr int rows(int form) { return form == VF_SEP ? SY : DY; }
};

// The copies of one window plane (NY x AX floats) that a thread issues: offsets
// within a slice and validity are the same for every slice of a segment.
template <int NY, int AX>
struct PlaneCopies {
    static constexpr int N16 = (NY * AX / 4 + NTHREADS - 1) / NTHREADS;
    int off[N16];        // 16-byte chunks: element offset in the slice; < 0: outside (zero)
    int y0, x0;          // the window's first row and column
    __device__ __forceinline__ void set(const VolJob& J, int y, int x) {
        y0 = y;
        x0 = x;
#pragma unroll
        for (int k = 0; k < N16; ++k) {
            const int c = threadIdx.x + k * NTHREADS, r = c / (AX / 4), gy = y + r, gx = x + 4 * (c - r * (AX / 4));
            const bool in = c < NY * AX / 4 && gy >= 0 && gy < J.h && gx >= 0 && gx < J.w;
            off[k] = in ? gy * J.w + gx : -1;  // a slice has fewer than 2^31 elements
        }
    }
    __device__ __forceinline__ void issue(const VolJob& J, const float* __restrict__ x, int z, float* A, bool vec) const {
        const unsigned int base = smem_u32(A);
        const bool zin = z >= 0 && z < J.d;
        const float* src = x + (long long)(zin ? z : 0) * J.h * J.w;
        if (vec) {
#pragma unroll
            for (int k = 0; k < N16; ++k) {
                const int c = threadIdx.x + k * NTHREADS;
                const bool in = zin && off[k] >= 0;
                if (c < NY * AX / 4)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(base + 16u * (unsigned int)c),
                                 "l"(in ? src + off[k] : x), "r"(in ? 16 : 0)
                                 : "memory");
            }
        } else {
            // a warp per row (rows start anywhere)
            const int lane = threadIdx.x & 31;
            for (int r = threadIdx.x >> 5; r < NY; r += NTHREADS / 32) {
                const int gy = y0 + r;
                const bool rin = zin && gy >= 0 && gy < J.h;
                const float* row = src + (long long)(rin ? gy : 0) * J.w;
#pragma unroll
                for (int c = lane; c < AX; c += 32) {
                    const int gx = x0 + c;
                    const bool in = rin && gx >= 0 && gx < J.w;
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                                     base + 4u * (unsigned int)(r * AX + c)),
                                 "l"(in ? row + gx : x), "r"(in ? 4 : 0)
                                 : "memory");
                }
            }
        }
    }
};

__device__ __forceinline__ void commit_copies() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void wait_copies() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ float elem(const float4& v, int k) {
    return k == 0 ? v.x : (k == 1 ? v.y : (k == 2 ? v.z : v.w));
}
__device__ __forceinline__ bool aligned16(const void* a, const void* b, const void* c) {
    return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(c)) & 15) == 0;
}

// One segment of a phase's range: slices z0 .. z1 - 1 of the tile at (y0, x0).
struct Segment {
    int y0, x0, z0, z1;
};
template <int SY>
__device__ __forceinline__ bool next_segment(const VolJob& J, long long& u, long long u_end, Segment& g) {
    if (u >= u_end) return false;
    const int ntx = (J.w + MX - 1) / MX, tile = (int)(u / J.d);
    g.z0 = (int)(u - (long long)tile * J.d);
    g.z1 = (int)min((long long)J.d, g.z0 + (u_end - u));
    g.x0 = (tile % ntx) * MX;
    g.y0 = (tile / ntx) * SY;
    u += g.z1 - g.z0;
    return true;
}
__device__ __forceinline__ long long tile_units(const VolJob& J, int sy) {
    return (long long)((J.w + MX - 1) / MX) * ((J.h + sy - 1) / sy) * J.d;
}

// One convolution phase of a separable PSF, out = epilogue(C (*) x).
template <int R>
__device__ __forceinline__ void sep_phase(const VolJob& J, const float* __restrict__ x, float* sm, const EpiArgs& E,
                                          DF (&acc)[2]) {
    using M = March<R>;
    constexpr int RPT = M::RPT, QX = M::QX, HQ = M::PADX / 4;
    const int tid = threadIdx.x, q = tid % QX, g = tid / QX;  // quad of the staged row, row group
    const bool work = g < M::GR, main = work && q >= HQ && q < QX - HQ;
    float* V = sm + M::RING * M::SPLANE;
    const long long units = tile_units(J, M::SY);
    long long u = units * blockIdx.x / gridDim.x;
    const long long u_end = units * (blockIdx.x + 1) / gridDim.x;
    const bool vin = (J.w & 3) == 0 && aligned16(x, nullptr, nullptr);
    const bool vec = (J.w & 3) == 0 && aligned16(E.a, E.b, E.out);
    const size_t sl = (size_t)J.h * J.w;
    PlaneCopies<M::SY + 2 * R, M::AX> P;
    Segment G;
    while (next_segment<M::SY>(J, u, u_end, G)) {
        const int gx = G.x0 + 4 * (q - HQ), gy = G.y0 + g * RPT;
        int nv[RPT];  // outputs of each row inside the volume (<= 0: none)
#pragma unroll
        for (int i = 0; i < RPT; ++i) nv[i] = main && gy + i < J.h ? min(4, J.w - gx) : 0;
        const int s0 = G.z0 - R, s_end = G.z1 + R;  // input slices
        P.set(J, G.y0 - R, G.x0 - M::PADX);
        __syncthreads();  // the ring and V of the segment before
#pragma unroll
        for (int k = 0; k < M::RING; ++k) {
            if (s0 + k < s_end) P.issue(J, x, s0 + k, sm + k * M::SPLANE, vin);
            commit_copies();
        }
        constexpr int NP = R > 0 ? 2 * R : 1;
        float4 part[RPT][NP];  // partial sums of the outputs s - R + k before slice s
#pragma unroll
        for (int i = 0; i < RPT; ++i)
#pragma unroll
            for (int k = 0; k < NP; ++k) part[i][k] = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 own[RPT];  // the finished slice's quads, waiting for the columns pass
        int slot = 0;
        size_t at = ((size_t)G.z0 * J.h + gy) * J.w + gx;
#pragma unroll 1
        for (int s = s0; s <= s_end; ++s, slot = (slot + 1) & (M::RING - 1)) {
            // the slice finished one step ago: z = s - 1 - R
            const bool emit = s - 1 - R >= G.z0;
            float4 pa[RPT], pb[RPT];
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                pa[i] = pb[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (emit && nv[i] > 0) {
                    // g is read once a solve: streaming, it leaves L2 to r
                    if (E.mode == VE_RESID && vec)
                        pa[i] = __ldcs(reinterpret_cast<const float4*>(E.a + at + (size_t)(i * J.w)));
                    else if (E.a)
                        pa[i] = ld_quad(E.a, at + (size_t)(i * J.w), nv[i], vec);
                    if (E.b) pb[i] = ld_quad(E.b, at + (size_t)(i * J.w), nv[i], vec);
                }
            }
            wait_copies<M::RING - 2>();  // plane s (and s + 1) has landed
            __syncthreads();             // V of slice s - 1 is complete; the slot of plane s - 1 is free
            if (s > s0) {
                if (s + M::RING - 1 < s_end)
                    P.issue(J, x, s + M::RING - 1, sm + ((slot + M::RING - 1) & (M::RING - 1)) * M::SPLANE, vin);
                commit_copies();
            }
            const int b = slot & 1;
            if (emit && main) {  // columns pass
                const float4* v = reinterpret_cast<const float4*>(V + (b ^ 1) * M::V) + g * RPT * QX + q;
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    float w[4 * (2 * HQ + 1)];
#pragma unroll
                    for (int j = 0; j <= 2 * HQ; ++j) {
                        const float4 t = j == HQ ? own[i] : v[i * QX + j - HQ];
                        w[4 * j] = t.x;
                        w[4 * j + 1] = t.y;
                        w[4 * j + 2] = t.z;
                        w[4 * j + 3] = t.w;
                    }
                    float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int k = 0; k <= 2 * R; ++k)
#pragma unroll
                        for (int c = 0; c < 4; ++c) o[c] = fmaf(J.taps.cx[k], w[M::PADX - R + c + k], o[c]);
                    if (nv[i] > 0)
                        epilogue4(E, at + (size_t)(i * J.w), nv[i], vec, make_float4(o[0], o[1], o[2], o[3]),
                                  pa[i], pb[i], acc);
                }
            }
            if (emit) at += sl;
            if (s < s_end && work) {  // rows pass, then along the slices
                const float4* a = reinterpret_cast<const float4*>(sm + slot * M::SPLANE) + g * RPT * QX + q;
                float4 h[RPT];
#pragma unroll
                for (int i = 0; i < RPT; ++i) h[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int p = 0; p < 2 * R + RPT; ++p) {
                    const float4 t = a[p * QX];
#pragma unroll
                    for (int i = 0; i < RPT; ++i)
                        if (p - i >= 0 && p - i <= 2 * R) h[i] = fma4(J.taps.cy[p - i], t, h[i]);
                }
                float4* v = reinterpret_cast<float4*>(V + b * M::V) + g * RPT * QX + q;
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    if constexpr (R == 0) {
                        own[i] = mul4(J.taps.cz[0], h[i]);
                    } else {
                        own[i] = fma4(J.taps.cz[2 * R], h[i], part[i][0]);
#pragma unroll
                        for (int k = 0; k < 2 * R - 1; ++k) part[i][k] = fma4(J.taps.cz[2 * R - 1 - k], h[i], part[i][k + 1]);
                        part[i][2 * R - 1] = mul4(J.taps.cz[0], h[i]);
                    }
                    v[i * QX] = own[i];
                }
            }
        }
    }
    wait_copies<0>();
}

// Four outputs from the tap list, in global memory: what rows of taps sum to where
// every voxel is finite.  A row's taps of weight zero would carry an infinite or NaN voxel
// (0 x inf) to outputs that no tap takes it to, so those outputs come from here.
template <int R>
__device__ __noinline__ float4 tap_sums(const VolJob& J, const float* __restrict__ x, int z, int y, int x0, int nv) {
    float o[4] = {0.f, 0.f, 0.f, 0.f};
    for (int k = 0; k < J.taps.ntap; ++k) {
        const int4 t = __ldg(J.gtaps + k);
        const int gz = z + t.x, gy = y + t.y;
        if (gz < 0 || gz >= J.d || gy < 0 || gy >= J.h) continue;
        const float* row = x + ((long long)gz * J.h + gy) * J.w;
        for (int i = 0; i < nv; ++i) {
            const int gx = x0 + i + t.z;
            if (gx >= 0 && gx < J.w) o[i] = fmaf(__int_as_float(t.w), __ldcg(row + gx), o[i]);
        }
    }
    return make_float4(o[0], o[1], o[2], o[3]);
}

// One convolution phase of a PSF with dense rows of taps.
template <int R>
__device__ __forceinline__ void dense_phase(const VolJob& J, const float* __restrict__ x, float* sm, const EpiArgs& E,
                                            DF (&acc)[2]) {
    using M = March<R>;
    const int tid = threadIdx.x, q = tid & 15, row = tid >> 4;  // four columns of one row
    float* W = sm + M::RING * M::DPLANE;                        // W[((dy + R) (2R + 1) + dz + R) 4 NW4 + dx + R]
    unsigned int* mask = reinterpret_cast<unsigned int*>(W + M::WTS);  // slice offsets with taps, by row offset
    const long long units = tile_units(J, M::DY);
    long long u = units * blockIdx.x / gridDim.x;
    const long long u_end = units * (blockIdx.x + 1) / gridDim.x;
    const bool vin = (J.w & 3) == 0 && aligned16(x, nullptr, nullptr);
    const bool vec = (J.w & 3) == 0 && aligned16(E.a, E.b, E.out);
    for (int i = tid; i < M::WTS; i += NTHREADS) W[i] = 0.f;
    if (tid < 16) mask[tid] = 0u;
    __syncthreads();
    for (int k = tid; k < J.taps.ntap; k += NTHREADS) {
        const int4 t = __ldg(J.gtaps + k);
        W[((t.y + R) * (2 * R + 1) + t.x + R) * (4 * M::NW4) + t.z + R] = __int_as_float(t.w);
        atomicOr(&mask[t.y + R], 1u << (t.x + R));
    }
    PlaneCopies<M::DY + 2 * R, M::AX> P;
    Segment G;
    while (next_segment<M::DY>(J, u, u_end, G)) {
        const int gx = G.x0 + 4 * q, gy = G.y0 + row;
        const int nv = gy < J.h ? min(4, J.w - gx) : 0;  // outputs inside the volume (<= 0: none)
        const int s0 = max(G.z0 - R, 0), s_end = min(G.z1 + R, J.d);  // input slices (those outside are zero)
        P.set(J, G.y0 - R, G.x0 - M::PADX);
        __syncthreads();  // the taps; the ring of the segment before
#pragma unroll
        for (int k = 0; k < M::RING; ++k) {
            if (s0 + k < s_end) P.issue(J, x, s0 + k, sm + k * M::DPLANE, vin);
            commit_copies();
        }
        float4 part[2 * R + 1];  // partial sums of the outputs z = s - R + k
#pragma unroll
        for (int k = 0; k <= 2 * R; ++k) part[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        int slot = 0;
#pragma unroll 1
        for (int s = s0; s < G.z1 + R; ++s, slot = (slot + 1) & (M::RING - 1)) {
            // the epilogue's operands of output slice s - R, fetched ahead
            const int z = s - R;
            const bool emit = z >= G.z0 && nv > 0;
            const size_t at = ((size_t)(z >= G.z0 ? z : G.z0) * J.h + gy) * J.w + gx;
            float4 pa = make_float4(0.f, 0.f, 0.f, 0.f), pb = pa;
            if (emit && E.a) pa = ld_quad(E.a, at, nv, vec);
            if (emit && E.b) pb = ld_quad(E.b, at, nv, vec);
            wait_copies<M::RING - 2>();  // plane s has landed
            __syncthreads();             // the slot of plane s - 1 is free
            if (s > s0) {
                if (s + M::RING - 1 < s_end)
                    P.issue(J, x, s + M::RING - 1, sm + ((slot + M::RING - 1) & (M::RING - 1)) * M::DPLANE, vin);
                commit_copies();
            }
            // slice offsets whose output lies in the segment: k = z - s + R for z in [z0, z1)
            const int k_lo = max(G.z0 - z, 0), k_hi = min(G.z1 - 1 - z, 2 * R);
            const unsigned int seg = s < s_end && k_lo <= k_hi ? ((2u << (2 * R - k_lo)) - 1u) & ~((1u << (2 * R - k_hi)) - 1u) : 0u;
            constexpr int NQ = (4 + 2 * M::PADX) / 4;
            const float* A = sm + slot * M::DPLANE;
#pragma unroll 1
            for (int p = 0; p <= 2 * R; ++p) {
                const unsigned int mk = mask[p] & seg;
                if (mk == 0u) continue;
                const float4* a = reinterpret_cast<const float4*>(A + (row + p) * M::AX) + q;
                float w[4 * NQ];
#pragma unroll
                for (int j = 0; j < NQ; ++j) {
                    const float4 v = a[j];
                    w[4 * j] = v.x;
                    w[4 * j + 1] = v.y;
                    w[4 * j + 2] = v.z;
                    w[4 * j + 3] = v.w;
                }
                const float4* Wp = reinterpret_cast<const float4*>(W) + p * (2 * R + 1) * M::NW4;
#pragma unroll
                for (int k = 0; k <= 2 * R; ++k) {  // slice offset R - k: output z = s - R + k
                    if ((mk >> (2 * R - k)) & 1u) {
#pragma unroll
                        for (int j = 0; j < M::NW4; ++j) {
                            const float4 t = Wp[(2 * R - k) * M::NW4 + j];
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (4 * j + e <= 2 * R) {
                                    constexpr int o = M::PADX - R;
                                    part[k].x = fmaf(elem(t, e), w[o + 4 * j + e], part[k].x);
                                    part[k].y = fmaf(elem(t, e), w[o + 1 + 4 * j + e], part[k].y);
                                    part[k].z = fmaf(elem(t, e), w[o + 2 + 4 * j + e], part[k].z);
                                    part[k].w = fmaf(elem(t, e), w[o + 3 + 4 * j + e], part[k].w);
                                }
                        }
                    }
                }
            }
            if (emit) {
                const float4 t = part[0];
                if (!isfinite((t.x + t.y) + (t.z + t.w))) part[0] = tap_sums<R>(J, x, z, gy, gx, nv);
                epilogue4(E, at, nv, vec, part[0], pa, pb, acc);
            }
#pragma unroll
            for (int k = 0; k < 2 * R; ++k) part[k] = part[k + 1];
            part[2 * R] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    wait_copies<0>();
}

// VF_SPARSE: few taps in a large support.  8 x 8 x 32 output tiles, staged with
// their halo; every output sums the tap list over the window.
template <int R>
struct SparseTile {
    static constexpr int NZ = TZ + 2 * R, NY = TY + 2 * R, AX = TX + 2 * R;
    static constexpr size_t bytes = sizeof(float) * (size_t)NZ * NY * AX;
};
template <int R>
__device__ __forceinline__ void sparse_phase(const VolJob& J, const float* __restrict__ x, float* A, const EpiArgs& E,
                                             DF (&acc)[2]) {
    using S = SparseTile<R>;
    const int ntx = (J.w + TX - 1) / TX, nty = (J.h + TY - 1) / TY;
    const int ntiles = ntx * nty * ((J.d + TZ - 1) / TZ);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned int base = smem_u32(A);
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int x0 = (t % ntx) * TX, y0 = ((t / ntx) % nty) * TY, z0 = (t / ntx / nty) * TZ;
        __syncthreads();
        for (int r = warp; r < S::NZ * S::NY; r += NTHREADS / 32) {
            const int gz = z0 - R + r / S::NY, gy = y0 - R + r % S::NY;
            const bool rin = gz >= 0 && gz < J.d && gy >= 0 && gy < J.h;
            const float* src = x + ((long long)(rin ? gz : 0) * J.h + (rin ? gy : 0)) * J.w;
            for (int c = lane; c < S::AX; c += 32) {
                const int gx = x0 - R + c;
                const bool in = rin && gx >= 0 && gx < J.w;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                                 base + 4u * (unsigned int)(r * S::AX + c)),
                             "l"(in ? src + gx : x), "r"(in ? 4 : 0)
                             : "memory");
            }
        }
        asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const int gx = x0 + lane, gy = y0 + warp;
        float s[TZ];
#pragma unroll
        for (int z = 0; z < TZ; ++z) s[z] = 0.f;
        const float* a = A + (R * S::NY + warp + R) * S::AX + lane + R;
        for (int k = 0; k < J.taps.ntap; ++k) {
            const int4 tp = __ldg(J.gtaps + k);
            const float* b = a + (tp.x * S::NY + tp.y) * S::AX + tp.z;
#pragma unroll
            for (int z = 0; z < TZ; ++z) s[z] = fmaf(__int_as_float(tp.w), b[z * S::NY * S::AX], s[z]);
        }
        if (gx < J.w && gy < J.h) {
#pragma unroll
            for (int z = 0; z < TZ; ++z) {
                if (z0 + z >= J.d) break;
                const size_t i = ((size_t)(z0 + z) * J.h + gy) * J.w + gx;
                E.out[i] = epilogue(E, s[z], E.a ? __ldcg(E.a + i) : 0.f, E.b ? __ldcg(E.b + i) : 0.f, acc);
            }
        }
    }
}

// VF_SMALL: 8 x 8 x 32 output tiles, the next tile's window (zero outside the
// volume) in flight by cp.async while this one is convolved: slices over every
// staged (row, column) into B, rows into C (over the window's own buffer),
// columns over C.  A marching block repeats 2 r slices whatever its share, so below
// 2 r slices a block the tiles are faster.  GB300, one convolution in tiles | marched, us:
// 45 x 70 x 61, r = 2 (0.4 slices a block) 4.7 | 5.8; 62 x 146 x 25, r = 3 (1.2) 5.0 | 13.3; 128^3
// (4.2 up to r = 4) r = 1 10.0 | 7.5, r = 2 11.8 | 10.8, r = 3 15.0 | 15.7, r = 4 16.0 | 21.2;
// 160^3, r = 3 (9.5) 27.2 | 21.9.  The line was drawn up to r = 4: with the 12-row tiles
// of r = 6 marching is ahead of it, 128^3 (9.3 slices a block) 44.1 | 28.6.
template <int R>
struct SmallTile {
    static constexpr int PADX = (R + 3) / 4 * 4, X0 = PADX - R;
    static constexpr int NZ = TZ + 2 * R, NY = TY + 2 * R, AX = TX + 2 * PADX;
    static constexpr int IN = NZ * NY * AX, MID = TZ * NY * AX;
    static constexpr size_t bytes = sizeof(float) * (2 * (size_t)IN + MID);
};
template <int R>
__device__ __forceinline__ void stage_small(const VolJob& J, const float* __restrict__ x, int x0, int y0, int z0, float* A,
                                            bool vec) {
    using S = SmallTile<R>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned int base = smem_u32(A);
    if (vec) {
        constexpr int CH = S::AX / 4, RPW = 32 / CH, ROWS = S::NZ * S::NY;  // chunks per row, rows per warp
        const int sub = lane / CH, c = lane - sub * CH;
        for (int r0 = warp * RPW; r0 < ROWS; r0 += (NTHREADS / 32) * RPW) {
            const int row = r0 + sub;
            if (sub >= RPW || row >= ROWS) continue;
            const int gz = z0 - R + row / S::NY, gy = y0 - R + row % S::NY, gx = x0 - S::PADX + 4 * c;
            const bool in = gz >= 0 && gz < J.d && gy >= 0 && gy < J.h && gx >= 0 && gx < J.w;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                             base + 4u * (unsigned int)(row * S::AX + 4 * c)),
                         "l"(in ? x + ((long long)gz * J.h + gy) * J.w + gx : x), "r"(in ? 16 : 0)
                         : "memory");
        }
    } else {
        for (int row = warp; row < S::NZ * S::NY; row += NTHREADS / 32) {
            const int gz = z0 - R + row / S::NY, gy = y0 - R + row % S::NY;
            const bool rin = gz >= 0 && gz < J.d && gy >= 0 && gy < J.h;
            const float* src = x + ((long long)(rin ? gz : 0) * J.h + (rin ? gy : 0)) * J.w;
#pragma unroll
            for (int c = lane; c < S::AX; c += 32) {
                const int gx = x0 - S::PADX + c;
                const bool in = rin && gx >= 0 && gx < J.w;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                                 base + 4u * (unsigned int)(row * S::AX + c)),
                             "l"(in ? src + gx : x), "r"(in ? 4 : 0)
                             : "memory");
            }
        }
    }
    commit_copies();
}
template <int R>
__device__ __forceinline__ void small_phase(const VolJob& J, const float* __restrict__ x, float* sm, const EpiArgs& E,
                                            DF (&acc)[2]) {
    using S = SmallTile<R>;
    const VolTaps& K = J.taps;
    const int ntx = (J.w + TX - 1) / TX, nty = (J.h + TY - 1) / TY;
    const int ntiles = ntx * nty * ((J.d + TZ - 1) / TZ), nb = gridDim.x;
    const int xo = threadIdx.x & 31, yo = threadIdx.x >> 5;
    const bool vec = (J.w & 3) == 0 && aligned16(x, nullptr, nullptr);
    float* B = sm + 2 * S::IN;
    int t = blockIdx.x, buf = 0;
    if (t >= ntiles) return;  // the whole block
    auto origin = [&](int k, int& x0, int& y0, int& z0) {
        x0 = (k % ntx) * TX;
        y0 = ((k / ntx) % nty) * TY;
        z0 = (k / ntx / nty) * TZ;
    };
    int x0, y0, z0;
    origin(t, x0, y0, z0);
    stage_small<R>(J, x, x0, y0, z0, sm, vec);
    for (; t < ntiles; t += nb, buf ^= 1) {
        origin(t, x0, y0, z0);
        if (t + nb < ntiles) {
            int x1, y1, z1;
            origin(t + nb, x1, y1, z1);
            stage_small<R>(J, x, x1, y1, z1, sm + (buf ^ 1) * S::IN, vec);
            wait_copies<1>();
        } else {
            wait_copies<0>();
        }
        __syncthreads();
        float* A = sm + buf * S::IN;
        const int gx = x0 + xo, gy = y0 + yo;
        const bool in = gy < J.h && gx < J.w;
        // the epilogue's operands, fetched before the passes
        float pa[TZ], pb[TZ];
#pragma unroll
        for (int z = 0; z < TZ; ++z) {
            const size_t i = ((size_t)(z0 + z) * J.h + gy) * J.w + gx;
            const bool ok = in && z0 + z < J.d;
            pa[z] = ok && E.a ? __ldcg(E.a + i) : 0.f;
            pb[z] = ok && E.b ? __ldcg(E.b + i) : 0.f;
        }
        constexpr int COLS = S::NY * S::AX;
        for (int c = threadIdx.x; c < COLS; c += NTHREADS) {
            float win[S::NZ];
#pragma unroll
            for (int z = 0; z < S::NZ; ++z) win[z] = A[z * COLS + c];
#pragma unroll
            for (int z = 0; z < TZ; ++z) {
                float s = 0.f;
#pragma unroll
                for (int o = 0; o <= 2 * R; ++o) s = fmaf(K.cz[o], win[z + o], s);
                B[z * COLS + c] = s;
            }
        }
        __syncthreads();
        constexpr int COLS2 = TZ * S::AX;
        for (int c = threadIdx.x; c < COLS2; c += NTHREADS) {
            const int z = c / S::AX, xx = c - z * S::AX;
            const float* b = B + z * COLS + xx;
            float win[S::NY];
#pragma unroll
            for (int y = 0; y < S::NY; ++y) win[y] = b[y * S::AX];
#pragma unroll
            for (int y = 0; y < TY; ++y) {
                float s = 0.f;
#pragma unroll
                for (int p = 0; p <= 2 * R; ++p) s = fmaf(K.cy[p], win[y + p], s);
                A[(z * TY + y) * S::AX + xx] = s;
            }
        }
        __syncthreads();
        float s[TZ];
#pragma unroll
        for (int z = 0; z < TZ; ++z) {
            s[z] = 0.f;
            const float* c = A + (z * TY + yo) * S::AX + S::X0 + xo;
#pragma unroll
            for (int q = 0; q <= 2 * R; ++q) s[z] = fmaf(K.cx[q], c[q], s[z]);
        }
        if (in) {
#pragma unroll
            for (int z = 0; z < TZ; ++z) {
                if (z0 + z >= J.d) break;
                E.out[((size_t)(z0 + z) * J.h + gy) * J.w + gx] = epilogue(E, s[z], pa[z], pb[z], acc);
            }
        }
        __syncthreads();  // the buffers are restaged after this
    }
}

template <int R>
__device__ __forceinline__ void conv_phase(const VolJob& J, const float* __restrict__ x, float* sm, const EpiArgs& E,
                                           DF (&acc)[2]) {
    if (J.taps.form == VF_SEP)
        sep_phase<R>(J, x, sm, E, acc);
    else if (J.taps.form == VF_SMALL)
        small_phase<R>(J, x, sm, E, acc);
    else if (J.taps.form == VF_DENSE)
        dense_phase<R>(J, x, sm, E, acc);
    else
        sparse_phase<R>(J, x, sm, E, acc);
}

// A vector phase over float4 elements i = gtid, gtid + gstr, ...: two elements
// per step, every load of both issued before the first store (the stores may
// alias nothing the loads need, but the compiler cannot prove it).
// f(x, y) maps the NL loaded values to the NS stored ones.  REV: from the last element
// to the first, so that a phase finds the end of what the phase before streamed still
// in L2 (the update after the new directions), and the first output streaming (u, not
// read again before the next update): 256^3, 3 iterations, 3.09 -> 3.03 GB of DRAM traffic
// by the order alone, 2.98 with u and g streamed.
template <bool REV, int NL, int NS, class F>
__device__ __forceinline__ void vec_phase(long long n4, long long gtid, long long gstr,
                                          const float4* const (&in)[NL], float4* const (&out)[NS],
                                          F&& f) {
    for (long long e = gtid; e < n4; e += 2 * gstr) {
        const bool second = e + gstr < n4;
        const long long i = REV ? n4 - 1 - e : e, j = REV ? i - gstr : i + gstr;
        float4 x0[NL], x1[NL], y[NS];
#pragma unroll
        for (int k = 0; k < NL; ++k) x0[k] = __ldcg(in[k] + i);
        if (second) {
#pragma unroll
            for (int k = 0; k < NL; ++k) x1[k] = __ldcg(in[k] + j);
        }
        f(x0, y);
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            if (REV && k == 0) __stcs(out[k] + i, y[k]);
            else out[k][i] = y[k];
        }
        if (second) {
            f(x1, y);
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                if (REV && k == 0) __stcs(out[k] + j, y[k]);
                else out[k][j] = y[k];
            }
        }
    }
}

// ------------------------------------------------------------- level solve

__device__ __forceinline__ bool pos_finite(double x) { return x > 0.0 && isfinite(x); }

// MR-II (the three-term recurrence of the oracle's level smoother):
//   r0 = g - H u0;  p1 = H r0, q1 = H p1, a = <r,q>/<q,q>, u += a p, r -= a q;
//   then while k < m and the stop test fails:
//   z = H q_k, b1 = <z,q_k>/<q_k,q_k>, b2 = <z,q_{k-1}>/<q_{k-1},q_{k-1}> (k >= 2),
//   q_{k+1} = z - b1 q_k - b2 q_{k-1}, p_{k+1} = q_k - b1 p_k - b2 p_{k-1},
//   a = <r,q_{k+1}>/<q_{k+1},q_{k+1}>, u += a p_{k+1}, r -= a q_{k+1}.
// p and q live in rings of three buffers: p_k = P[(k - 1) % 3].  The phases run in
// one loop with one convolution, one update and one reduction in the code: on the
// small levels a phase's first execution is bound by the fetch of its instructions.
enum VolPhase : int { PH_ZERO = 0, PH_R0, PH_P1, PH_Q1, PH_Z, PH_DIR, PH_UPD };

template <int R>
__global__ void __launch_bounds__(NTHREADS, 2) k_vol_mr2(const __grid_constant__ VolJob J) {
    extern __shared__ __align__(16) float sm[];
    __shared__ VolScal S;
    const unsigned int nb = gridDim.x, bid = blockIdx.x;
    const long long gtid = (long long)bid * NTHREADS + threadIdx.x, gstr = (long long)nb * NTHREADS;
    float4* u4 = reinterpret_cast<float4*>(J.u);
    float4* r4 = reinterpret_cast<float4*>(J.R);
    {
        // the vector phases run on whole float4s: zero the (at most 3) padding
        // voxels past n of every vector this solve reads, whatever an earlier
        // use of the shared buffers left there
        const long long pad = 4 * J.n4 - J.n;
        if (gtid < pad) {
            const long long i = J.n + gtid;
            J.u[i] = 0.f;
            J.R[i] = 0.f;
            J.Z[i] = 0.f;
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                J.P[b][i] = 0.f;
                J.Q[b][i] = 0.f;
            }
        }
    }
    unsigned int phase = 0;
    bool ok = true;
    int kind = J.zero_start ? PH_ZERO : PH_R0;
#pragma unroll 1
    for (;;) {
        DF acc[2] = {{0.f, 0.f}, {0.f, 0.f}};
        const int k = kind >= PH_Z ? S.k : 0;  // PH_Z, PH_DIR: from q_k to q_{k+1}; PH_UPD: applies step k + 1
        const int cur = (k + 2) % 3, prv = (k + 1) % 3, nxt = k % 3;  // buffers of steps k, k - 1, k + 1
        if (kind == PH_DIR) {
            // q_{k+1}, p_{k+1}; <q_{k+1}, q_{k+1}>, <r, q_{k+1}>
            const float b1 = S.b1, b2 = S.b2;
            float4* const out[2] = {reinterpret_cast<float4*>(J.Q[nxt]), reinterpret_cast<float4*>(J.P[nxt])};
            if (k >= 2) {
                const float4* const in[6] = {reinterpret_cast<const float4*>(J.Z),
                                             reinterpret_cast<const float4*>(J.Q[cur]),
                                             reinterpret_cast<const float4*>(J.P[cur]), r4,
                                             reinterpret_cast<const float4*>(J.Q[prv]),
                                             reinterpret_cast<const float4*>(J.P[prv])};
                vec_phase<false, 6, 2>(J.n4, gtid, gstr, in, out, [&](const float4 (&x)[6], float4 (&y)[2]) {
                    y[0] = fma4(-b2, x[4], fma4(-b1, x[1], x[0]));
                    y[1] = fma4(-b2, x[5], fma4(-b1, x[2], x[1]));
                    acc_add(acc[0], dot4(y[0], y[0], 0.f));
                    acc_add(acc[1], dot4(x[3], y[0], 0.f));
                });
            } else {
                const float4* const in[4] = {reinterpret_cast<const float4*>(J.Z),
                                             reinterpret_cast<const float4*>(J.Q[cur]),
                                             reinterpret_cast<const float4*>(J.P[cur]), r4};
                vec_phase<false, 4, 2>(J.n4, gtid, gstr, in, out, [&](const float4 (&x)[4], float4 (&y)[2]) {
                    y[0] = fma4(-b1, x[1], x[0]);
                    y[1] = fma4(-b1, x[2], x[1]);
                    acc_add(acc[0], dot4(y[0], y[0], 0.f));
                    acc_add(acc[1], dot4(x[3], y[0], 0.f));
                });
            }
        } else if (kind == PH_UPD) {
            // u += a p_{k+1}, r -= a q_{k+1}; ||r||^2
            const float a = S.a;
            const float4* const in[4] = {reinterpret_cast<const float4*>(J.P[nxt]),
                                         reinterpret_cast<const float4*>(J.Q[nxt]), u4, r4};
            float4* const out[2] = {u4, r4};
            vec_phase<true, 4, 2>(J.n4, gtid, gstr, in, out, [&](const float4 (&x)[4], float4 (&y)[2]) {
                y[0] = fma4(a, x[0], x[2]);
                y[1] = fma4(-a, x[1], x[3]);
                acc_add(acc[0], dot4(y[1], y[1], 0.f));
            });
        } else if (kind == PH_ZERO) {
            // a zero start: u = 0, r = g
            const float4* g4 = reinterpret_cast<const float4*>(J.g);
            for (long long i = gtid; i < J.n4; i += gstr) {
                const float4 g = __ldcg(g4 + i);
                u4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                r4[i] = g;
                acc_add(acc[0], dot4(g, g, 0.f));
            }
            acc[1] = acc[0];
        } else {
            // r0 = g - H u0 | p1 = H r0 | q1 = H p1 | z = H q_k, with the sums each needs
            const float* x = kind == PH_R0 ? J.u : (kind == PH_P1 ? J.R : (kind == PH_Q1 ? J.P[0] : J.Q[cur]));
            EpiArgs E;
            E.mode = kind - PH_R0 + VE_RESID;
            E.a = kind == PH_R0 ? J.g : (kind == PH_P1 ? nullptr : (kind == PH_Q1 ? J.R : J.Q[cur]));
            E.b = kind == PH_Z && k >= 2 ? J.Q[prv] : nullptr;
            E.out = kind == PH_R0 ? J.R : (kind == PH_P1 ? J.P[0] : (kind == PH_Q1 ? J.Q[0] : J.Z));
            conv_phase<R>(J, x, sm, E, acc);
        }
        ok = grid_reduce_df<2>(acc, J.partials, J.gs, nb, bid, phase++, [&](const DF (&t)[2]) {
            const double t0 = df_to_double(t[0]), t1 = df_to_double(t[1]);
            if (kind <= PH_R0) {
                S.rr = t0;
                S.k = 0;
                // the limit of both rules, formed once (off the later phases' path)
                S.lim2 = fmax(J.conv_tol > 0.0 ? J.conv_tol * J.conv_tol * t1 : -1.0,
                              J.stop_tol > 0.0 ? J.stop_tol * J.stop_tol * (double)J.n : -1.0);
                S.done = (J.m <= 0 || t0 <= S.lim2) ? 1 : 0;
            } else if (kind == PH_Q1 || kind == PH_DIR) {
                S.done = pos_finite(t0) ? 0 : 2;
                S.qqn = t0;
                S.a = (float)(t1 / t0);
            } else if (kind == PH_Z) {
                S.b1 = (float)(t0 / S.qq);
                S.b2 = k >= 2 ? (float)(t1 / S.qqp) : 0.f;
            } else if (kind == PH_UPD) {
                S.rr = t0;
                S.qqp = S.qq;
                S.qq = S.qqn;
                S.k = k + 1;
                S.done = (S.k >= J.m || t0 <= S.lim2) ? 1 : 0;
            }
        });
        if (!ok || S.done) break;
        kind = kind == PH_ZERO || kind == PH_R0 ? PH_P1
               : kind == PH_P1                  ? PH_Q1
               : kind == PH_Q1 || kind == PH_DIR ? PH_UPD
               : kind == PH_UPD                 ? PH_Z
                                                : PH_DIR;
    }
    if (bid == 0 && threadIdx.x == 0) {
        J.out[0] = S.k;
        J.out[1] = S.rr;
        J.out[2] = ok ? S.done : -1;
    }
    grid_exit(J.gs, nb);
}

// H x (or H^T x with the transposed taps) of a whole level.
template <int R>
__global__ void __launch_bounds__(NTHREADS, 2) k_vol_apply(const __grid_constant__ VolJob J,
                                                           const float* __restrict__ x, float* __restrict__ y) {
    extern __shared__ __align__(16) float sm[];
    DF acc[2] = {{0.f, 0.f}, {0.f, 0.f}};
    conv_phase<R>(J, x, sm, EpiArgs{nullptr, nullptr, y, VE_STORE}, acc);
}

// Shared memory of the solve and apply kernels of radius r, and the rows of the
// tiles whose slices a phase divides over the blocks.
template <int R>
constexpr size_t vol_smem(int form) {
    return form == VF_SPARSE ? SparseTile<R>::bytes : form == VF_SMALL ? SmallTile<R>::bytes : March<R>::bytes(form);
}
template <int R>
constexpr int vol_tile_rows(int form) {
    return March<R>::rows(form);
}

// The solve and apply kernels of radius r (0 .. EECMG_VOL_MAX_RADIUS), from the
// translation unit that instantiates them; false if r is outside its range.
bool vol_kernels_r012(int r, const void** solve, const void** apply);
bool vol_kernels_r34(int r, const void** solve, const void** apply);
bool vol_kernels_r56(int r, const void** solve, const void** apply);

}  // namespace vol
}  // namespace eecmg
