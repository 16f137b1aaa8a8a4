// level_start.cuh -- the start of a prolonged level (Algorithm 2, Step 2),
// D(S(P(Pi(u1, u2)))), one warp per strip of columns marching down the rows.
//
// The operator chain is instruction-bound (S alone takes eight weights, nine moments
// and an elimination per pixel), so the kernel is built to issue few
// instructions per pixel and to need no barrier:
//   - a lane owns one level-(l-2) cell: 4 fine columns, two level-(l-1) columns
//     and one node; Pi's node differences, its double-float sums and P's column
//     rule are evaluated once per level-(l-1) row, not once per fine pixel;
//   - every stage keeps the rows it needs in registers (P two rows, S three,
//     c two) and takes the one column beyond its own from the neighbouring lane;
//   - a weight of S belongs to a pair of pixels and is computed once for both
//     where both are the lane's own (4.75 exponentials per pixel instead of 8),
//     and so is a flux of D.
// A 128-column strip yields the 116 columns of lanes 1..29 (S, c and D each
// consume one column per side, and lane 31 lacks its right-hand node), a segment
// of n rows computes n + 6.  The arithmetic per pixel is that of k_prolong,
// k_smooth and k_denoise (bitwise), so a result does not depend on the split.
//
// GB300, one start (32 x 64 tiles staged in shared memory before -> this): 4096^2 312
// -> 161 us, 2048^2 88 -> 49 us, 64^2 19 -> 11 us; its 88 MB at 4096^2 would take 13 us, so
// it stays bound by the issue of its instructions (22 us of the 161 are the exponentials'
// subnormal results, 16 the correctly rounded reciprocals).
#pragma once

#include "level_ops.cuh"

namespace eecmg {

constexpr int ST_WARPS = 4;               // warps (strip segments) per block
// Blocks per SM: three leave 168 registers a thread and nothing spills; four (128
// registers, 68 bytes spilled) gained 2 % at 4096^2 and lost 10 % at 2048^2, 20 % below.
constexpr int ST_MINB = 3;
constexpr int ST_CELLS = 29;              // cells a strip yields
constexpr int ST_COLS = 4 * ST_CELLS;     // 116 fine columns

struct StartArgs {
    const float* u1;
    const float* u2;
    float* out;
    int h1, w1, h2, w2, h, w;
    float scale, tau, ik2;
};

// EDGE: the strip touches the left or right edge of the image (columns outside
// it carry no weight, flux or store).
template <bool EDGE>
__device__ __forceinline__ void start_strip(const StartArgs& A, int strip, int ys, int ye) {
    const unsigned int FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int B = strip * ST_CELLS - 1 + lane, x = 4 * B;
    const int h = A.h, w = A.w, h1 = A.h1, w1 = A.w1, w2 = A.w2;
    const float ks = s_scale_ks(A.scale), tau = A.tau, ik2 = A.ik2;
    // v[k]: column x - 1 + k lies in the image (k = 0 the left neighbour's column, 5 the right one's)
    bool v[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = !EDGE || (x - 1 + k >= 0 && x - 1 + k < w);
    const bool node_r = B + 1 <= w2 - 1;   // the odd column's second node exists
    const bool col_b = 2 * B + 1 <= w1 - 1, col_c = 2 * B + 2 <= w1 - 1;
    const float* p1a = A.u1 + min(max(2 * B, 0), w1 - 1);
    const float* p1b = A.u1 + min(max(2 * B + 1, 0), w1 - 1);
    const float* p2 = A.u2 + min(max(B, 0), w2 - 1);

    // Pi's value from the centre and a quarter of the mean node difference
    auto pi = [](float u, DF d, float f) {
        const DF e = df_add2(DF{u, 0.f}, DF{__fmul_rn(f, d.hi), __fmul_rn(f, d.lo)});
        return __fadd_rn(e.hi, e.lo);
    };
    // P along the columns: the lane's four fine columns of one level-(l-1) row
    auto columns = [&](float xa, float xb, float (&H)[4]) {
        if (!col_b) xb = xa;
        float xc = __shfl_down_sync(FULL, xa, 1);
        if (!col_c) xc = xb;
        H[0] = xa;
        H[1] = __fmaf_rn(-0.125f, xc, __fmaf_rn(0.75f, xb, __fmul_rn(0.375f, xa)));
        H[2] = xb;
        H[3] = __fmaf_rn(0.375f, xc, __fmaf_rn(0.75f, xb, __fmul_rn(-0.125f, xa)));
    };
    // the node differences d(A, B) and the sum with the next node, d(A, B) + d(A, B + 1)
    auto nodes = [&](float u1v, float u2v, DF& d, DF& e) {
        d = two_sum(u1v, -u2v);
        const DF r{__shfl_down_sync(FULL, d.hi, 1), __shfl_down_sync(FULL, d.lo, 1)};
        e = df_add2(d, node_r ? r : d);
    };

    const int y0 = max(ys - 3, 0);
    int cell = y0 >> 2;
    DF dA, eA;          // nodes of the cell's first row
    float H[3][4];      // P along the columns at level-(l-1) rows 2 cell, + 1, + 2 (clamped)
    {
        const float a = p1a[(size_t)(2 * cell) * w1], b = p1b[(size_t)(2 * cell) * w1];
        nodes(a, p2[(size_t)cell * w2], dA, eA);
        columns(pi(a, dA, 0.25f), pi(b, eA, 0.125f), H[2]);
    }
    // the operands of the next cell row, fetched one cell row ahead
    float n1a, n1b, n2a, n2b, nu2;
    auto fetch = [&](int c) {
        const size_t r1 = (size_t)min(2 * c + 1, h1 - 1) * w1, r2 = (size_t)min(2 * c + 2, h1 - 1) * w1;
        n1a = p1a[r1];
        n1b = p1b[r1];
        n2a = p1a[r2];
        n2b = p1b[r2];
        nu2 = p2[(size_t)min(c + 1, A.h2 - 1) * w2];
    };
    fetch(cell);

    float Pp[6];                       // P, the row before
    SRow top[4];                       // the weights from the row before into it
    float Sm[6], Sp[4];                // S, one row (with neighbours) and two rows before
    float Cp[4], part[4];              // c and the first three fluxes of D, two rows before
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        top[c] = SRow{0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        Sp[c] = Cp[c] = part[c] = 0.f;
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) Pp[k] = Sm[k] = 0.f;
    const bool vec = (w & 3) == 0 && (reinterpret_cast<uintptr_t>(A.out) & 15) == 0;

#pragma unroll 1
    for (int y = y0; y < ye + 3; ++y) {
        float Pn[6];
        const bool row = y < h;
        if (row) {
            if (y == y0 || (y & 3) == 0) {  // enter cell row y / 4
                const bool has1 = 2 * cell + 1 <= h1 - 1, has2 = 2 * cell + 2 <= h1 - 1;
                DF dN = dA, eN = eA;
                if (has2) nodes(n2a, nu2, dN, eN);
#pragma unroll
                for (int c = 0; c < 4; ++c) H[0][c] = H[1][c] = H[2][c];
                if (has1) {
                    columns(pi(n1a, df_add2(dA, dN), 0.125f), pi(n1b, df_add2(eA, eN), 0.0625f), H[1]);
#pragma unroll
                    for (int c = 0; c < 4; ++c) H[2][c] = H[1][c];
                }
                if (has2) columns(pi(n2a, dN, 0.25f), pi(n2b, eN, 0.125f), H[2]);
                dA = dN;
                eA = eN;
                ++cell;
                fetch(cell);
            }
            const int ty = y & 3;
            const float q0 = c_qw[ty][0], q1 = c_qw[ty][1], q2 = c_qw[ty][2];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                Pn[c + 1] = __fmaf_rn(q2, H[2][c], __fmaf_rn(q1, H[1][c], __fmul_rn(q0, H[0][c])));
                if (EDGE && !v[c + 1]) Pn[c + 1] = 0.f;
            }
            Pn[0] = __shfl_up_sync(FULL, Pn[4], 1);
            Pn[5] = __shfl_down_sync(FULL, Pn[1], 1);
        } else {
#pragma unroll
            for (int k = 0; k < 6; ++k) Pn[k] = 0.f;
        }

        // the pairs between rows y - 1 and y: vert[c] in column c, diag[k] from column
        // k - 1 above to k below, anti[k] from column k above to k - 1 below
        SRow bot[4], topn[4];
        if (row && y > y0) {
            float vt[4], vtv[4], dg[5], dgv[5], an[5], anv[5];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float d = __fadd_rn(Pn[c + 1], -Pp[c + 1]);
                vt[c] = s_weight(d, ks);
                vtv[c] = __fmul_rn(vt[c], d);
            }
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const bool in = k == 0 ? v[0] : v[k + 1];
                const float d = __fadd_rn(Pn[k + 1], -Pp[k]), a = __fadd_rn(Pn[k], -Pp[k + 1]);
                dg[k] = s_weight(d, ks);
                an[k] = s_weight(a, ks);
                if (EDGE && !in) dg[k] = an[k] = 0.f;
                dgv[k] = __fmul_rn(dg[k], d);
                anv[k] = __fmul_rn(an[k], a);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                bot[c] = s_row(an[c], vt[c], dg[c + 1], anv[c], vtv[c], dgv[c + 1]);
                topn[c] = s_row(dg[c], vt[c], an[c + 1], -dgv[c], -vtv[c], -anv[c + 1]);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) bot[c] = topn[c] = SRow{0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        }

        // S of row y - 1
        float Sn[6];
        {
            float hz[5], hzv[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const float d = __fadd_rn(Pp[k + 1], -Pp[k]);
                hz[k] = s_weight(d, ks);
                if (EDGE && !(k == 0 ? v[0] : v[k + 1])) hz[k] = 0.f;
                hzv[k] = __fmul_rn(hz[k], d);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c)
                Sn[c + 1] = s_value(Pp[c + 1], top[c], bot[c], hz[c], hz[c + 1], -hzv[c], hzv[c + 1]);
            Sn[0] = __shfl_up_sync(FULL, Sn[4], 1);
            Sn[5] = __shfl_down_sync(FULL, Sn[1], 1);
        }

        // c of row r = y - 2, its fluxes along the row, the flux from row r into r - 1, D of row r - 1
        const int r = y - 2;
        float C[6], E[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float uc = Sm[c + 1];
            C[c + 1] = pm_c_value(v[c + 2] ? Sm[c + 2] : uc, (c > 0 || v[0]) ? Sm[c] : uc, r + 1 < h ? Sn[c + 1] : uc,
                                  r > 0 ? Sp[c] : uc, ik2);
        }
        C[5] = __shfl_down_sync(FULL, C[1], 1);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            E[c] = pm_flux(C[c + 1], C[c + 2], Sm[c + 1], Sm[c + 2]);
            if (EDGE && !v[c + 2]) E[c] = 0.f;
        }
        float E0 = __shfl_up_sync(FULL, E[3], 1);
        if (EDGE && !v[0]) E0 = 0.f;
        float o[4];
        const bool vert = r >= 1 && r < h;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float f = vert ? pm_flux(Cp[c], C[c + 1], Sp[c], Sm[c + 1]) : 0.f;
            o[c] = __fmaf_rn(tau, __fadd_rn(part[c], f), Sp[c]);
            part[c] = __fadd_rn(__fadd_rn(E[c], -(c == 0 ? E0 : E[c - 1])), -f);
            Cp[c] = C[c + 1];
            Sp[c] = Sm[c + 1];
            top[c] = topn[c];
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            Sm[k] = Sn[k];
            Pp[k] = Pn[k];
        }
        const int ro = y - 3;
        if (ro >= ys && lane >= 1 && lane <= ST_CELLS) {
            float* dst = A.out + (size_t)ro * w + x;
            if (vec) {
                if (!EDGE || x < w) *reinterpret_cast<float4*>(dst) = make_float4(o[0], o[1], o[2], o[3]);
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (!EDGE || v[c + 1]) dst[c] = o[c];
            }
        }
    }
}

// One warp's unit of the level: segment `unit / strips` (th rows) of strip `unit % strips`.
__device__ __forceinline__ void start_unit(const StartArgs& A, int strips, int th, int unit) {
    const int strip = unit % strips, ys = (unit / strips) * th;
    if (ys >= A.h) return;  // the whole warp
    const int ye = min(ys + th, A.h);
    const int x_end = 4 * (strip * ST_CELLS - 1 + 32) + 1;  // one past the strip's last column and its neighbour
    if (strip == 0 || x_end > A.w)
        start_strip<true>(A, strip, ys, ye);
    else
        start_strip<false>(A, strip, ys, ye);
}

}  // namespace eecmg
