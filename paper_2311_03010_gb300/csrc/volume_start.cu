// volume_start.cu -- the operators that start a level of the volume cascade:
// the new extrapolation Pi and quadratic interpolation P (Section 3.2 per
// axis), local smoothing S (Section 3.3) and the Perona-Malik step D
// (Section 4), each in one pass over its output.
//
// A thread owns a column (Pi, P: a cell of a column) and marches along the
// slices, so that what a slice contributes to its neighbours is formed once
// and kept in registers; in-slice neighbours come from shared-memory planes.
// GB300 at 256^3, one voxel per thread before -> now: Pi (128^3) 19 -> 11 us, P
// 206 -> 18 us (its taps came from a per-lane constant index), S 825 -> 245 us, D
// 140 -> 70 us (134 + 201 MB: at the memory's rate).
#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "volume_start.hpp"

namespace eecmg {
namespace vol {

namespace {

constexpr int SMS = 152;

// Slices per block of a marching kernel: enough blocks for six per SM, between
// lo (each block repeats two slices' work) and 32.
int slices_per_block(int d, long long columns, int lo) {
    const long long n = ((long long)d * columns + 6 * SMS - 1) / (6 * SMS);
    return (int)std::min<long long>(32, std::max<long long>(lo, n));
}

// ------------------------------------------------------------------ Pi, P

// Pi: u1 + (1/4) x the mean of the level-(l-2) differences over the cell's
// eight corners (indices past the last level-(l-2) node clamp to it).  A thread
// takes column b of a node cell: the sums over the cell's four (slice, row)
// nodes of d(., B0) + d(., B1) serve its 2 x 2 outputs.
constexpr int PX = 32, PY = 8;
__global__ void __launch_bounds__(PX * PY) k_vol_pi(const float* __restrict__ u1, int d1, int h1, int w1,
                                                    const float* __restrict__ u2, int d2, int h2, int w2,
                                                    float* __restrict__ out) {
    const int b = blockIdx.x * PX + (threadIdx.x & (PX - 1)), A = blockIdx.y * PY + threadIdx.x / PX, C = blockIdx.z;
    if (b >= w1 || A >= h2) return;
    const int B0 = b >> 1, B1 = (b & 1) ? min(B0 + 1, w2 - 1) : B0;
    const int As[2] = {A, min(A + 1, h2 - 1)}, Cs[2] = {C, min(C + 1, d2 - 1)};
    float e[2][2];
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const float* p1 = u1 + ((long long)(2 * Cs[x]) * h1 + 2 * As[y]) * w1;
            const float* p2 = u2 + ((long long)Cs[x] * h2 + As[y]) * w2;
            e[x][y] = (__ldg(p1 + 2 * B0) - __ldg(p2 + B0)) + (__ldg(p1 + 2 * B1) - __ldg(p2 + B1));
        }
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const int c = 2 * C + x, a = 2 * A + y;
            if (c >= d1 || a >= h1) continue;
            const float s = (e[0][0] + e[0][y]) + (e[x][0] + e[x][y]);
            const long long v = ((long long)c * h1 + a) * w1 + b;
            out[v] = fmaf(0.03125f, s, __ldg(u1 + v));
        }
}

// P: the three-point Lagrange rule at offsets 0, 1/4, 1/2, 3/4 of a level-(l-2)
// cell along every axis (clamped indices).  A thread takes one output column of
// a cell and its 4 x 4 outputs in (slice, row): the columns are interpolated
// once per coarse row (9), the rows once per coarse slice.
__global__ void __launch_bounds__(PX * PY) k_vol_quad(const float* __restrict__ ut, int d1, int h1, int w1,
                                                      float* __restrict__ out, int d, int h, int w) {
    const int x = blockIdx.x * PX + (threadIdx.x & (PX - 1)), Y = blockIdx.y * PY + threadIdx.x / PX, Z = blockIdx.z;
    if (x >= w || 4 * Y >= h) return;
    const int tx = x & 3, X = (x >> 2) * 2;
    const float q0 = tx == 0 ? 1.f : (tx == 1 ? 0.375f : (tx == 2 ? 0.f : -0.125f));
    const float q1 = tx == 0 ? 0.f : (tx == 2 ? 1.f : 0.75f);
    const float q2 = tx == 1 ? -0.125f : (tx == 3 ? 0.375f : 0.f);
    const int x1 = min(X + 1, w1 - 1), x2 = min(X + 2, w1 - 1);
    float r[3][4];
#pragma unroll
    for (int o = 0; o < 3; ++o) {
        float c[3];
#pragma unroll
        for (int p = 0; p < 3; ++p) {
            const float* row = ut + ((long long)min(2 * Z + o, d1 - 1) * h1 + min(2 * Y + p, h1 - 1)) * w1;
            c[p] = fmaf(q2, __ldg(row + x2), fmaf(q1, __ldg(row + x1), q0 * __ldg(row + X)));
        }
        r[o][0] = c[0];
        r[o][1] = fmaf(-0.125f, c[2], fmaf(0.75f, c[1], 0.375f * c[0]));
        r[o][2] = c[1];
        r[o][3] = fmaf(0.375f, c[2], fmaf(0.75f, c[1], -0.125f * c[0]));
    }
    float* o = out + ((long long)(4 * Z) * h + 4 * Y) * w + x;
    const long long sl = (long long)h * w;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (4 * Y + i >= h) break;
        o[0] = r[0][i];
        if (4 * Z + 1 < d) o[sl] = fmaf(-0.125f, r[2][i], fmaf(0.75f, r[1][i], 0.375f * r[0][i]));
        if (4 * Z + 2 < d) o[2 * sl] = r[1][i];
        if (4 * Z + 3 < d) o[3 * sl] = fmaf(0.375f, r[2][i], fmaf(0.75f, r[1][i], -0.125f * r[0][i]));
        o += w;
    }
}

// ----------------------------------------------------------------------- S

constexpr int SX = 32, SY = 8, SN = (SX + 2) * (SY + 2);  // a plane with its halo

// Weighted sums over one slice of the 3 x 3 x 3 neighbourhood (offsets s along
// the rows, t along the columns; v = neighbour - centre).
struct Plane {
    float w, ws, wt, wss, wtt, wst, v, vs, vt;
};

// p: the slice's nine values; MID: the centre's own slice (its centre has weight
// 1 and v = 0, added by the caller).  EDGE: `in` bit 3 (s + 1) + t + 1 says that
// the (s, t) neighbour lies in the volume.
template <bool MID, bool EDGE>
__device__ __forceinline__ Plane plane_sums(const float (&p)[9], float uc, float ks, unsigned int in) {
    float wl[3], wc[3], wr[3], vl[3], vc[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        float wt[3], v[3];
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            const bool ctr = MID && s == 1 && t == 1;
            v[t] = ctr ? 0.f : p[3 * s + t] - uc;
            const float e = v[t] * ks;
            wt[t] = ctr ? 0.f : ex2_approx(-e * e);
            if (EDGE && !((in >> (3 * s + t)) & 1u)) wt[t] = 0.f;
        }
        wl[s] = wt[2] - wt[0];          // first moment along the row
        wr[s] = wt[2] + wt[0];          // second
        wc[s] = wr[s] + wt[1];          // weight
        const float a = wt[0] * v[0];
        vl[s] = fmaf(wt[2], v[2], -a);
        vc[s] = fmaf(wt[2], v[2], a);
        if (!(MID && s == 1)) vc[s] = fmaf(wt[1], v[1], vc[s]);
    }
    Plane r;
    r.wss = wc[0] + wc[2];
    r.w = r.wss + wc[1];
    r.ws = wc[2] - wc[0];
    r.wt = (wl[0] + wl[2]) + wl[1];
    r.wtt = (wr[0] + wr[2]) + wr[1];
    r.wst = wl[2] - wl[0];
    r.v = (vc[0] + vc[2]) + vc[1];
    r.vs = vc[2] - vc[0];
    r.vt = (vl[0] + vl[2]) + vl[1];
    return r;
}

// The fitted value: raw moments, centred at the end (offsets in {-1, 0, 1} and a
// centre of weight 1: a centred diagonal moment is at least 1/27 of the raw one),
// then slope . ob = c^T C^+ ob by elimination, pivots of at most 1e-6 W dropped.
// A direction of small variance lambda carries c' and ob' of order lambda, so
// its whole term is of that order: whether a pivot or an eigenvalue meets the
// cut changes the value by about 1e-6 of a neighbour difference.
__device__ __forceinline__ float fit_value(float uc, const Plane& T, const Plane& M, const Plane& B) {
    const float m00 = T.w + B.w, W = (m00 + M.w) + 1.f;
    const float o0 = B.w - T.w, o1 = (T.ws + B.ws) + M.ws, o2 = (T.wt + B.wt) + M.wt;
    const float m11 = (T.wss + B.wss) + M.wss, m22 = (T.wtt + B.wtt) + M.wtt, m12 = (T.wst + B.wst) + M.wst;
    const float m01 = B.ws - T.ws, m02 = B.wt - T.wt;
    const float c0 = B.v - T.v, c1 = (T.vs + B.vs) + M.vs, c2 = (T.vt + B.vt) + M.vt, sv = (T.v + B.v) + M.v;
    const float iw = recip(W), b0 = o0 * iw, b1 = o1 * iw, b2 = o2 * iw, vb = sv * iw, thr = 1e-6f * W;
    const float a00 = fmaf(-b0, o0, m00), a01 = fmaf(-b0, o1, m01), a02 = fmaf(-b0, o2, m02);
    const float a11 = fmaf(-b1, o1, m11), a12 = fmaf(-b1, o2, m12), a22 = fmaf(-b2, o2, m22);
    const float k0 = fmaf(-vb, o0, c0), k1 = fmaf(-vb, o1, c1), k2 = fmaf(-vb, o2, c2);
    const float r0 = a00 > thr ? recip(a00) : 0.f;
    const float l1 = a01 * r0, l2 = a02 * r0;
    const float d1 = fmaf(-l1, a01, a11), e1 = fmaf(-l1, a02, a12);
    const float k1p = fmaf(-l1, k0, k1), b1p = fmaf(-l1, b0, b1);
    const float r1 = d1 > thr ? recip(d1) : 0.f;
    const float l3 = e1 * r1;
    const float d2 = fmaf(-l3, e1, fmaf(-l2, a02, a22));
    const float k2p = fmaf(-l3, k1p, fmaf(-l2, k0, k2)), b2p = fmaf(-l3, b1p, fmaf(-l2, b0, b2));
    const float r2 = d2 > thr ? recip(d2) : 0.f;
    const float g = fmaf(k0 * b0, r0, fmaf(k1p * b1p, r1, (k2p * b2p) * r2));
    return (uc + vb) - g;
}

// S: per voxel the weighted hyperplane fit over the in-volume 3 x 3 x 3
// neighbourhood, weights exp(-(scale v)^2).  Bound by instruction issue: 26
// exponentials of four instructions and 464 instructions in all per voxel (256^3: 245 us, issuing
// 87 % of the time; 825 us with the eigen-decomposition that this elimination replaced).
template <bool EDGE>
__device__ __forceinline__ void smooth_column(float (&A)[2][SN], const float* __restrict__ u, int d, int h, int w,
                                              float ks, float* __restrict__ out, int z0, int z1, int x0, int y0) {
    const int tid = threadIdx.x, tx = tid & (SX - 1), ty = tid / SX, x = x0 + tx, y = y0 + ty;
    const long long sl = (long long)h * w;
    // the plane's elements this thread stages (clamped into the volume: what lies outside has no weight)
    const int e0 = tid, e1 = tid + SX * SY;
    auto src = [&](int e) {
        const int r = e / (SX + 2), c = e - r * (SX + 2);
        return (long long)min(max(y0 - 1 + r, 0), h - 1) * w + min(max(x0 - 1 + c, 0), w - 1);
    };
    const long long g0 = src(e0), g1 = src(min(e1, SN - 1));
    unsigned int in = 0;  // in-plane neighbours inside the volume
    if (EDGE) {
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int yy = y + k / 3 - 1, xx = x + k % 3 - 1;
            if (yy >= 0 && yy < h && xx >= 0 && xx < w) in |= 1u << k;
        }
    }
    float f0, f1 = 0.f;
    auto fetch = [&](int z) {
        const float* p = u + sl * min(max(z, 0), d - 1);
        f0 = __ldg(p + g0);
        if (e1 < SN) f1 = __ldg(p + g1);
    };
    int buf = 0;
    auto stage = [&](float (&P)[9]) {  // the fetched plane to shared memory, its 3 x 3 window to registers
        A[buf][e0] = f0;
        if (e1 < SN) A[buf][e1] = f1;
        __syncthreads();
        const float* a = A[buf] + ty * (SX + 2) + tx;
#pragma unroll
        for (int k = 0; k < 9; ++k) P[k] = a[(k / 3) * (SX + 2) + k % 3];
        buf ^= 1;
    };
    float P0[9], P1[9], P2[9];  // slices z - 1, z, z + 1
    fetch(z0 - 1);
    stage(P0);
    fetch(z0);
    stage(P1);
    fetch(z0 + 1);
    float* dst = out + (long long)y * w + x;
#pragma unroll 1
    for (int z = z0; z < z1; ++z) {
        stage(P2);
        fetch(z + 2);
        const float uc = P1[4];
        Plane T{}, B{};
        if (z > 0) T = plane_sums<false, EDGE>(P0, uc, ks, in);
        const Plane M = plane_sums<true, EDGE>(P1, uc, ks, in);
        if (z + 1 < d) B = plane_sums<false, EDGE>(P2, uc, ks, in);
        if (!EDGE || (x < w && y < h)) dst[sl * z] = fit_value(uc, T, M, B);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            P0[k] = P1[k];
            P1[k] = P2[k];
        }
    }
}

__global__ void __launch_bounds__(SX * SY, 3) k_vol_smooth(const float* __restrict__ u, int d, int h, int w, float ks,
                                                          float* __restrict__ out, int zc) {
    __shared__ float A[2][SN];
    const int x0 = blockIdx.x * SX, y0 = blockIdx.y * SY, z0 = blockIdx.z * zc, z1 = min(z0 + zc, d);
    if (x0 > 0 && y0 > 0 && x0 + SX < w && y0 + SY < h)
        smooth_column<false>(A, u, d, h, w, ks, out, z0, z1, x0, y0);
    else
        smooth_column<true>(A, u, d, h, w, ks, out, z0, z1, x0, y0);
}

// ----------------------------------------------------------------------- D

// D: u' = u + tau x sum over in-volume face neighbours of (c_nb + c) / 2 (u_nb - u),
// c = 1 / (1 + |grad u|^2 / k^2) with central differences (an out-of-volume
// neighbour replaced by the centre): a pass for c and one for the step.  A thread
// owns four columns of a row and marches along the slices (its own slices and
// the flux between them in registers, column neighbours by shuffles in groups
// of 16 lanes), so a pass loads three float4 per operand and four voxels.  One
// fused pass (c in shared memory) was tried: its halo and barriers cost more
// (115 us at 256^3) than the c volume's round trip through L2.
constexpr int DX = 64, DY = 16;
// Four columns of a row from p; VEC: 16-byte aligned, else nv of them exist and
// the rest read as the last.
template <bool VEC>
__device__ __forceinline__ void ld4v(const float* __restrict__ p, int nv, float (&o)[4]) {
    if (VEC) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(p));
        o[0] = v.x;
        o[1] = v.y;
        o[2] = v.z;
        o[3] = v.w;
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k] = __ldg(p + min(k, nv - 1));
    }
}
template <bool VEC>
__device__ __forceinline__ void st4v(float* p, int nv, const float (&o)[4]) {
    if (VEC) {
        *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < nv) p[k] = o[k];
    }
}
// A thread's place: columns x .. x + nv - 1 of row y; offsets in a slice of its row
// and of the rows before and after it (clamped: the thread's own row at the
// volume's edge), and of the columns beyond its 16-lane group.
struct Place {
    int own, north, south, west, east, nv;
    bool active, first, last;
};
__device__ __forceinline__ Place place(int h, int w) {
    const int t = threadIdx.x & 15, x = blockIdx.x * DX + 4 * t, y = blockIdx.y * DY + (threadIdx.x >> 4);
    Place P;
    P.active = x < w && y < h;
    const int xc = P.active ? x : 0, yc = P.active ? y : 0;
    P.nv = min(4, w - xc);
    P.own = yc * w + xc;
    P.north = P.own - (yc > 0 ? w : 0);
    P.south = P.own + (yc + 1 < h ? w : 0);
    P.west = P.own - (xc > 0 ? 1 : 0);
    P.east = P.own + min(4, w - 1 - xc);
    P.first = t == 0;
    P.last = t == 15 || x + 4 >= w;
    return P;
}
// columns x - 1 .. x + 4: the thread's own and its neighbours' (an end of the row: the centre's own value)
__device__ __forceinline__ void row6(const float* __restrict__ s, const Place& P, const float (&v)[4], float (&o)[6]) {
    o[0] = __shfl_up_sync(0xffffffffu, v[3], 1, 16);
    o[5] = __shfl_down_sync(0xffffffffu, v[0], 1, 16);
    if (P.first) o[0] = __ldg(s + P.west);
    if (P.last) o[5] = __ldg(s + P.east);
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k + 1] = v[k];
}

template <bool VEC>
__global__ void __launch_bounds__(16 * DY) k_vol_pm_c(const float* __restrict__ u, int d, int h, int w, float ik2,
                                                      float* __restrict__ c, int zc) {
    const Place P = place(h, w);
    const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, d);
    const long long sl = (long long)h * w;
    const float* s = u + sl * z0;
    float* dst = c + sl * z0 + P.own;
    float ub[4], uc[4], un[4], nn[4], ss[4], r[6], o[4];
    ld4v<VEC>((z0 > 0 ? s - sl : s) + P.own, P.nv, ub);
    ld4v<VEC>(s + P.own, P.nv, uc);
#pragma unroll 1
    for (int z = z0; z < z1; ++z, s += sl, dst += sl) {
        ld4v<VEC>((z + 1 < d ? s + sl : s) + P.own, P.nv, un);
        ld4v<VEC>(s + P.north, P.nv, nn);
        ld4v<VEC>(s + P.south, P.nv, ss);
        row6(s, P, uc, r);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float gx = 0.5f * (r[k + 2] - r[k]), gy = 0.5f * (ss[k] - nn[k]), gz = 0.5f * (un[k] - ub[k]);
            o[k] = recip_ge1(fmaf(fmaf(gz, gz, fmaf(gx, gx, gy * gy)), ik2, 1.f));
            ub[k] = uc[k];
            uc[k] = un[k];
        }
        if (P.active) st4v<VEC>(dst, P.nv, o);
    }
}

template <bool VEC>
__global__ void __launch_bounds__(16 * DY) k_vol_pm_step(const float* __restrict__ u, const float* __restrict__ c, int d,
                                                         int h, int w, float tau, float* __restrict__ out, int zc) {
    const Place P = place(h, w);
    const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, d);
    const long long sl = (long long)h * w;
    const float *us = u + sl * z0, *cs = c + sl * z0;
    float* dst = out + sl * z0 + P.own;
    const float ht = 0.5f * tau;
    float uc[4], cc[4], un[4], cn[4], a[4], b[4], r[6], q[6], o[4], fb[4];
    ld4v<VEC>(us + P.own, P.nv, uc);
    ld4v<VEC>(cs + P.own, P.nv, cc);
    ld4v<VEC>((z0 > 0 ? us - sl : us) + P.own, P.nv, un);
    ld4v<VEC>((z0 > 0 ? cs - sl : cs) + P.own, P.nv, cn);
#pragma unroll
    for (int k = 0; k < 4; ++k) fb[k] = (cn[k] + cc[k]) * (uc[k] - un[k]);  // twice the flux into the slice before
#pragma unroll 1
    for (int z = z0; z < z1; ++z, us += sl, cs += sl, dst += sl) {
        // a neighbour beyond the volume reads as the centre: no flux
        ld4v<VEC>((z + 1 < d ? us + sl : us) + P.own, P.nv, un);
        ld4v<VEC>((z + 1 < d ? cs + sl : cs) + P.own, P.nv, cn);
        row6(us, P, uc, r);
        row6(cs, P, cc, q);
        float e = (q[0] + q[1]) * (r[1] - r[0]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float er = (q[k + 1] + q[k + 2]) * (r[k + 2] - r[k + 1]), f = (cc[k] + cn[k]) * (un[k] - uc[k]);
            o[k] = (er - e) + (f - fb[k]);
            e = er;
            fb[k] = f;
        }
        ld4v<VEC>(us + P.north, P.nv, a);
        ld4v<VEC>(cs + P.north, P.nv, b);
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k] = fmaf(b[k] + cc[k], a[k] - uc[k], o[k]);
        ld4v<VEC>(us + P.south, P.nv, a);
        ld4v<VEC>(cs + P.south, P.nv, b);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            o[k] = fmaf(ht, fmaf(b[k] + cc[k], a[k] - uc[k], o[k]), uc[k]);
            uc[k] = un[k];
            cc[k] = cn[k];
        }
        if (P.active) st4v<VEC>(dst, P.nv, o);
    }
}

unsigned int blocks(int n, int per) { return (unsigned int)((n + per - 1) / per); }

}  // namespace

cudaError_t launch_vol_pi(const float* u1, int d1, int h1, int w1, const float* u2, int d2, int h2, int w2,
                          float* out, cudaStream_t s) {
    k_vol_pi<<<dim3(blocks(w1, PX), blocks(h2, PY), d2), PX * PY, 0, s>>>(u1, d1, h1, w1, u2, d2, h2, w2, out);
    return cudaGetLastError();
}

cudaError_t launch_vol_quad(const float* ut, int d1, int h1, int w1, float* out, int d, int h, int w,
                            cudaStream_t s) {
    k_vol_quad<<<dim3(blocks(w, PX), blocks(h, 4 * PY), blocks(d, 4)), PX * PY, 0, s>>>(ut, d1, h1, w1, out, d, h, w);
    return cudaGetLastError();
}

cudaError_t launch_vol_smooth(const float* u, int d, int h, int w, float scale, float* out, cudaStream_t s) {
    const dim3 g(blocks(w, SX), blocks(h, SY));
    const int zc = slices_per_block(d, (long long)g.x * g.y, 4);
    k_vol_smooth<<<dim3(g.x, g.y, blocks(d, zc)), SX * SY, 0, s>>>(u, d, h, w, s_scale_ks(scale), out, zc);
    return cudaGetLastError();
}

cudaError_t launch_vol_denoise(const float* u, int d, int h, int w, float ik2, float tau, float* c, float* out,
                               cudaStream_t s) {
    const dim3 g(blocks(w, DX), blocks(h, DY));
    const int zc = slices_per_block(d, (long long)g.x * g.y, 2);
    const dim3 grid(g.x, g.y, blocks(d, zc));
    const uintptr_t all = reinterpret_cast<uintptr_t>(u) | reinterpret_cast<uintptr_t>(c) | reinterpret_cast<uintptr_t>(out);
    if ((w & 3) == 0 && (all & 15) == 0) {
        k_vol_pm_c<true><<<grid, 16 * DY, 0, s>>>(u, d, h, w, ik2, c, zc);
        k_vol_pm_step<true><<<grid, 16 * DY, 0, s>>>(u, c, d, h, w, tau, out, zc);
    } else {
        k_vol_pm_c<false><<<grid, 16 * DY, 0, s>>>(u, d, h, w, ik2, c, zc);
        k_vol_pm_step<false><<<grid, 16 * DY, 0, s>>>(u, c, d, h, w, tau, out, zc);
    }
    return cudaGetLastError();
}

}  // namespace vol
}  // namespace eecmg
