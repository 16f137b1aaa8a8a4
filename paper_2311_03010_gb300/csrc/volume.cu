// volume.cu -- EECMG on volumes (Algorithm 2 with every operator carried over
// to three dimensions; the paper names volumes as the method's next
// application without writing the 3-D operators out).
//
// The slice axis is treated exactly like the row and column axes:
//   restriction  coarse (a, b, c) = fine (2a, 2b, 2c)                (Eqs. 12-13)
//   H_l          zero-boundary 3-D convolution, K_l(o,p,q) = rho K(2o,2p,2q),
//                rho = N_{l+1} / N_l                                  (Eq. 14)
//   Pi           u^{l-1} + 1/4 of the trilinear interpolant of the level-(l-2)
//                differences                                         (Section 3.2)
//   P            the three-point quadratic rule along all three axes (Section 3.2)
//   S            weighted hyperplane fit over the 3x3x3 neighbourhood with the
//                Eq. 18 weights, elimination on the 3x3 moment matrix
//                (pivots of at most 1e-6 W dropped)                  (Section 3.3)
//   D            one explicit Perona-Malik step with six face neighbours
//                                                                    (Section 4)
//   C_l^m        MR-II with the discrepancy stop of Section 2 and m_l as its cap.
//
// GPU design.  A volume of d x h x w voxels is stored slice-major, x[(k h + i)
// w + j]; every level vector of the workspace is padded with zeros to a
// multiple of 4 voxels so the vector phases run on float4.  Each level solve is
// ONE cooperative launch (all blocks co-resident): its phases are separated by
// the grid barrier with the fused deterministic reduction of persistent.cuh
// (every block sums all blocks' partials in a fixed order and keeps its own
// replica of the scalars), so the m_l iterations never return to the host and
// the stop decision is taken on the device.  The convolution phases march tiles
// of columns along the slices from a ring of staged planes (the level solve is in
// volume_impl.cuh).  The level start (Pi, P, S, D) is a chain of kernels in
// volume_start.cu.  The cascade is captured once as a CUDA graph.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "plan.hpp"
#include "volume_impl.cuh"
#include "volume_start.hpp"

namespace eecmg {
namespace vol {

// Voxel kernels run on a 3-D grid of 32 x 8 blocks: x = column, y = row,
// z = slice (no index division).
constexpr int VBX = 32, VBY = 8;

#define VOXEL_INDEX(d, h, w)                                          \
    const int j = blockIdx.x * VBX + (threadIdx.x & (VBX - 1));       \
    const int i = blockIdx.y * VBY + (threadIdx.x / VBX);             \
    const int k = blockIdx.z;                                         \
    if (j >= (w) || i >= (h)) return;                                 \
    const long long v = ((long long)k * (h) + i) * (w) + j;

__global__ void __launch_bounds__(VBX * VBY) k_vol_restrict(const float* __restrict__ f, int hf, int wf,
                                                            float* __restrict__ c, int dc, int hc, int wc) {
    VOXEL_INDEX(dc, hc, wc)
    c[v] = f[((long long)(2 * k) * hf + 2 * i) * wf + 2 * j];
}

}  // namespace vol
}  // namespace eecmg

// ====================================================================== host

using namespace eecmg;
using namespace eecmg::vol;

struct eecmg_vol_s {
    int W = 0, H = 0, D = 0, L = 0;
    double tau = 0.2, kpm = 10.0;
    eecmg_options opt{};
    int device = 0, sms = 0;
    std::vector<int> ds, hs, ws, m;
    std::vector<long long> n, n4;
    std::vector<VolTaps> taps, tapsT;                  // H_l and H_l^T
    std::vector<std::vector<int4>> gt, gtT;            // general-form tap lists (host)
    char* wsp = nullptr;
    size_t ws_bytes = 0;
    std::vector<float*> g, u;                          // per level (padded)
    float* vec[8] = {};                                // R, P0..2, Q0..2, Z (finest size)
    int4* dtaps = nullptr;                             // all tap lists, [2l] H, [2l+1] H^T
    std::vector<size_t> dtap_off;
    GroupSync* gs = nullptr;                           // one per level
    double* partials = nullptr;
    double* out = nullptr;                             // 4 doubles per level
    std::vector<int> grid;                             // level solve blocks
    cudaStream_t cap = nullptr;
    cudaGraphExec_t gexec = nullptr;
    // optional per-launch timing (eager launches with an event pair around
    // each level start and each level solve)
    bool prof = false;
    std::vector<cudaEvent_t> ev;  // [4l .. 4l+3]: start begin/end, solve begin/end
    std::vector<int> ev_used;
};

namespace {

#define VCK(call)                                                                           \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess)                                                              \
            return set_error(EECMG_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

// Correlation-form taps of the PSF K (kd x kh x kw): C(d) = K(-d) for H,
// C(d) = K(d) for H^T.  A PSF that is an outer product of three vectors (to
// FP64 rounding) is stored as its three factors.
void make_vol_taps(const std::vector<double>& K, int kd, int kh, int kw, bool transpose,
                   VolTaps* t, std::vector<int4>* list) {
    std::memset(t, 0, sizeof(VolTaps));
    const int rz = kd / 2, ry = kh / 2, rx = kw / 2;
    const int r = std::max(rz, std::max(ry, rx));
    t->r = r;
    auto C = [&](int o, int p, int q) {
        if (!transpose) { o = -o; p = -p; q = -q; }
        return K[((size_t)(o + rz) * kh + (p + ry)) * kw + (q + rx)];
    };
    int o0 = 0, p0 = 0, q0 = 0;
    double mx = -1.0;
    for (int o = -rz; o <= rz; ++o)
        for (int p = -ry; p <= ry; ++p)
            for (int q = -rx; q <= rx; ++q)
                if (std::fabs(C(o, p, q)) > mx) {
                    mx = std::fabs(C(o, p, q));
                    o0 = o;
                    p0 = p;
                    q0 = q;
                }
    bool sep = mx > 0.0;
    if (sep) {
        // C(o,p,q) = a(o) b(p) c(q) through the largest entry k0:
        // a(o) = C(o,p0,q0), b(p) = C(o0,p,q0) / k0, c(q) = C(o0,p0,q) / k0
        const double k0 = C(o0, p0, q0);
        std::vector<double> a(kd), b(kh), c(kw);
        for (int o = -rz; o <= rz; ++o) a[o + rz] = C(o, p0, q0);
        for (int p = -ry; p <= ry; ++p) b[p + ry] = C(o0, p, q0) / k0;
        for (int q = -rx; q <= rx; ++q) c[q + rx] = C(o0, p0, q) / k0;
        for (int o = -rz; o <= rz && sep; ++o)
            for (int p = -ry; p <= ry && sep; ++p)
                for (int q = -rx; q <= rx; ++q)
                    if (std::fabs(C(o, p, q) - a[o + rz] * b[p + ry] * c[q + rx]) > 1e-12 * mx) {
                        sep = false;
                        break;
                    }
        if (sep) {
            for (int o = 0; o < kd; ++o) t->cz[o - rz + r] = (float)a[o];
            for (int p = 0; p < kh; ++p) t->cy[p - ry + r] = (float)b[p];
            for (int q = 0; q < kw; ++q) t->cx[q - rx + r] = (float)c[q];
        }
    }
    list->clear();
    if (!sep) {
        for (int o = -rz; o <= rz; ++o)
            for (int p = -ry; p <= ry; ++p)
                for (int q = -rx; q <= rx; ++q) {
                    const double v = C(o, p, q);
                    if (v == 0.0) continue;
                    float f = (float)v;
                    int bits;
                    std::memcpy(&bits, &f, 4);
                    // offsets into the staged tile relative to the output voxel
                    list->push_back(make_int4(o, p, q, bits));
                }
    }
    t->ntap = (int)list->size();
    // Rows of 2 r + 1 taps cost (2 r + 1) multiplications per row that holds a tap, on
    // register windows; a list costs a shared-memory read and a tap fetch per tap.  Up to
    // four times the multiplications the rows win (5^3 full support, 96 x 121 x 150: 13 us a
    // convolution against 157 us for the list).
    std::vector<char> row((size_t)kd * kh, 0);
    for (const int4& e : *list) row[(size_t)(e.x + rz) * kh + (e.y + ry)] = 1;
    const int rows = (int)std::count(row.begin(), row.end(), 1);
    t->form = sep ? VF_SEP : (rows * (2 * r + 1) <= 4 * t->ntap ? VF_DENSE : VF_SPARSE);
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Shared memory and tile rows of the kernels of radius r applying a PSF in `form`.
template <int R = VR>
size_t form_bytes(int r, int form) {
    if constexpr (R > 0)
        if (r < R) return form_bytes<R - 1>(r, form);
    return vol_smem<R>(form);
}
template <int R = VR>
int form_rows(int r, int form) {
    if constexpr (R > 0)
        if (r < R) return form_rows<R - 1>(r, form);
    return vol_tile_rows<R>(form);
}

// The kernels of every radius 0 .. EECMG_VOL_MAX_RADIUS (instantiated in the
// volume_r*.cu translation units).
struct VolKernels {
    const void* solve[VR + 1];
    const void* apply[VR + 1];
};
const VolKernels& vol_kernels() {
    static_assert(VR == 6, "instantiate every radius");
    static const VolKernels k = [] {
        VolKernels t{};
        for (int r = 0; r <= VR; ++r)
            if (!vol_kernels_r012(r, &t.solve[r], &t.apply[r]) &&
                !vol_kernels_r34(r, &t.solve[r], &t.apply[r]))
                vol_kernels_r56(r, &t.solve[r], &t.apply[r]);
        return t;
    }();
    return k;
}

// The 3-D grid of the voxel kernels for a d x h x w volume.
dim3 vgrid(int d, int h, int w) { return dim3((w + VBX - 1) / VBX, (h + VBY - 1) / VBY, d); }
constexpr int VTHREADS = VBX * VBY;

VolJob make_job(eecmg_vol_s* P, int l, bool transpose) {
    VolJob J{};
    J.d = P->ds[l];
    J.h = P->hs[l];
    J.w = P->ws[l];
    J.n = P->n[l];
    J.n4 = P->n4[l];
    J.g = P->g[l];
    J.u = P->u[l];
    J.R = P->vec[0];
    for (int i = 0; i < 3; ++i) {
        J.P[i] = P->vec[1 + i];
        J.Q[i] = P->vec[4 + i];
    }
    J.Z = P->vec[7];
    J.taps = transpose ? P->tapsT[l] : P->taps[l];
    J.gtaps = P->dtaps + P->dtap_off[2 * l + (transpose ? 1 : 0)];
    // general-form offsets index the staged tile: (dz + rz) NY AX + ...; the
    // kernel adds the output's own position, so store dz, dy, dx as they are
    J.m = P->m[l];
    J.stop_tol = P->opt.stop == EECMG_STOP_DISCREPANCY ? P->opt.c * P->opt.delta : 0.0;
    J.conv_tol = P->opt.conv_tol;
    J.partials = P->partials;
    J.gs = P->gs + l;
    J.out = P->out + 4 * l;
    return J;
}

// The (tile, slice) pairs a convolution phase divides over the blocks.
long long level_units(int d, int h, int w, const VolTaps& t) {
    if (t.form == VF_SMALL || t.form == VF_SPARSE)  // output tiles
        return (long long)((w + TX - 1) / TX) * ((h + TY - 1) / TY) * ((d + TZ - 1) / TZ);
    const int sy = form_rows(t.r, t.form);
    return (long long)((w + MX - 1) / MX) * ((h + sy - 1) / sy) * d;
}

eecmg_status launch_solve(eecmg_vol_s* P, int l, bool zero_start, cudaStream_t s) {
    VolJob J = make_job(P, l, false);
    J.zero_start = zero_start ? 1 : 0;
    void* args[] = {&J};
    const size_t smem = form_bytes(J.taps.r, J.taps.form);
    VCK(cudaLaunchCooperativeKernel(vol_kernels().solve[J.taps.r], dim3(P->grid[l]), dim3(NTHREADS),
                                    args, smem, s));
    return EECMG_OK;
}

eecmg_status launch_apply(eecmg_vol_s* P, int l, bool transpose, const float* x, float* y,
                          cudaStream_t s) {
    VolJob J = make_job(P, l, transpose);
    const size_t smem = form_bytes(J.taps.r, J.taps.form);
    const float* xx = x;
    void* args[] = {&J, (void*)&xx, (void*)&y};
    VCK(cudaLaunchKernel(vol_kernels().apply[J.taps.r], dim3((unsigned int)std::min<long long>(level_units(J.d, J.h, J.w, J.taps), 2 * P->sms)), dim3(NTHREADS),
                         args, smem, s));
    return EECMG_OK;
}

// D(S(P(Pi(u1, u2)))) of level l (l >= 2) into out; uses R, Z, P0, Q0 as
// temporaries (none of them is live between level solves).
eecmg_status launch_start(eecmg_vol_s* P, int l, const float* u1, const float* u2, float* out,
                          cudaStream_t s) {
    const int d1 = P->ds[l - 1], h1 = P->hs[l - 1], w1 = P->ws[l - 1];
    const int d = P->ds[l], h = P->hs[l], w = P->ws[l];
    float* ue = P->vec[4];   // Q0: Pi on level l-1
    float* ut = P->vec[0];   // R: P(Pi)
    float* sa = P->vec[1];   // P0
    float* cc = P->vec[7];   // Z: diffusivity
    VCK(launch_vol_pi(u1, d1, h1, w1, u2, P->ds[l - 2], P->hs[l - 2], P->ws[l - 2], ue, s));
    VCK(launch_vol_quad(ue, d1, h1, w1, ut, d, h, w, s));
    const int steps = P->opt.diffusion_steps;
    float* cur = steps == 0 ? out : sa;
    VCK(launch_vol_smooth(ut, d, h, w, (float)P->opt.s_scale, cur, s));
    const float ik2 = (float)(1.0 / (P->kpm * P->kpm));
    for (int st = 0; st < steps; ++st) {
        float* nxt = st == steps - 1 ? out : (cur == sa ? ut : sa);
        VCK(launch_vol_denoise(cur, d, h, w, ik2, (float)P->tau, cc, nxt, s));
        cur = nxt;
    }
    return EECMG_OK;
}

eecmg_status cascade(eecmg_vol_s* P, cudaStream_t s) {
    const int L = P->L;
    auto mark = [&](int l, int which) -> eecmg_status {
        if (!P->prof) return EECMG_OK;
        VCK(cudaEventRecord(P->ev[4 * l + which], s));
        P->ev_used[4 * l + which] = 1;
        return EECMG_OK;
    };
    for (int l = L - 1; l > 0; --l) {
        k_vol_restrict<<<vgrid(P->ds[l - 1], P->hs[l - 1], P->ws[l - 1]), VTHREADS, 0, s>>>(P->g[l], P->hs[l], P->ws[l],
                                                             P->g[l - 1], P->ds[l - 1],
                                                             P->hs[l - 1], P->ws[l - 1]);
        VCK(cudaGetLastError());
    }
    for (int l = 0; l < L; ++l) {
        eecmg_status st;
        if (l >= 2) {
            if ((st = mark(l, 0)) != EECMG_OK) return st;
            st = launch_start(P, l, P->u[l - 1], P->u[l - 2], P->u[l], s);
            if (st != EECMG_OK) return st;
            if ((st = mark(l, 1)) != EECMG_OK) return st;
        }
        if ((st = mark(l, 2)) != EECMG_OK) return st;
        st = launch_solve(P, l, l < 2, s);
        if (st != EECMG_OK) return st;
        if ((st = mark(l, 3)) != EECMG_OK) return st;
    }
    return EECMG_OK;
}

// Algorithmic bytes of level l's solve from the iterations it ran (each
// operand read or written once per phase, FP32): r0 12 per voxel; p1 = H r 8;
// q1 = H p with <r, q> 12; the first update 24; then per iteration k >= 1:
// z = H q_k with <z, q_k> (and <z, q_{k-1}> for k >= 2) 8 (12), the new
// directions 24 (32), the update 24.  A breakdown ends a level after the
// phase that found it.
double solve_bytes(const eecmg_vol_s* P, int l, int k, int reason) {
    double b = 12.0;
    const bool ran_first = k >= 1 || reason == 2;
    if (ran_first) b += 8.0 + 12.0;
    if (k >= 1) b += 24.0;
    for (int j = 1; j < k; ++j) b += (j >= 2 ? 12.0 : 8.0) + (j >= 2 ? 32.0 : 24.0) + 24.0;
    if (k >= 1 && reason == 2) b += (k >= 2 ? 12.0 : 8.0) + (k >= 2 ? 32.0 : 24.0);
    return b * (double)P->n[l];
}

// The cascade on the workspace's g_L (filled by the caller), as one CUDA graph
// captured at the first call (use_graph) or as plain launches.
eecmg_status run_cascade(eecmg_vol_s* P, cudaStream_t s) {
    if (!P->opt.use_graph || P->prof) return cascade(P, s);
    if (!P->gexec) {
        VCK(cudaStreamBeginCapture(P->cap, cudaStreamCaptureModeThreadLocal));
        eecmg_status st = cascade(P, P->cap);
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamEndCapture(P->cap, &graph);
        if (st != EECMG_OK) {
            if (graph) cudaGraphDestroy(graph);
            return st;
        }
        if (e != cudaSuccess)
            return set_error(EECMG_ERR_CUDA, std::string("volume graph capture: ") + cudaGetErrorString(e));
        e = cudaGraphInstantiate(&P->gexec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            P->gexec = nullptr;
            return set_error(EECMG_ERR_CUDA, std::string("volume graph instantiate: ") + cudaGetErrorString(e));
        }
    }
    VCK(cudaGraphLaunch(P->gexec, s));
    return EECMG_OK;
}

eecmg_status check_level(eecmg_vol_s* P, int level, const char* who) {
    if (!P) return set_error(EECMG_ERR_INVALID_ARG, std::string(who) + ": NULL plan");
    if (level < 0 || level >= P->L)
        return set_error(EECMG_ERR_INVALID_ARG, std::string(who) + ": level out of range");
    return EECMG_OK;
}

}  // namespace

extern "C" {

eecmg_status eecmg_vol_plan(int width, int height, int depth, int levels, const double* psf,
                            int psf_w, int psf_h, int psf_d, double alpha, double k,
                            const int* iters, const eecmg_options* opt, eecmg_vol_t* out) {
    if (!out) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_plan: out is NULL");
    *out = nullptr;
    if (width < 1 || height < 1 || depth < 1 || levels < 1 || levels > 16)
        return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_plan: bad volume size or levels");
    if ((long long)width * height * depth > (1LL << 31) || depth > 65535)
        return set_error(EECMG_ERR_INVALID_ARG,
                         "eecmg_vol_plan: volume above 2^31 voxels or 65535 slices");
    if (!psf || psf_w < 1 || psf_h < 1 || psf_d < 1 || !(psf_w & 1) || !(psf_h & 1) || !(psf_d & 1) ||
        psf_w / 2 > VR || psf_h / 2 > VR || psf_d / 2 > VR)
        return set_error(EECMG_ERR_INVALID_ARG,
                         "eecmg_vol_plan: PSF sides must be odd with radius <= EECMG_VOL_MAX_RADIUS");
    if (!(alpha >= 0.0 && alpha <= 0.25) || !(k > 0.0))
        return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_plan: need 0 <= alpha <= 0.25 and k > 0");
    eecmg_options o;
    eecmg_default_options(&o);
    if (opt) o = *opt;
    if (o.smoother != EECMG_SMOOTHER_MR2 || o.prolong != EECMG_PROLONG_EECMG ||
        o.storage != EECMG_STORAGE_FP32 || !o.workspace)
        return set_error(EECMG_ERR_UNSUPPORTED,
                         "eecmg_vol_plan: volumes run MR-II, Algorithm 2, FP32, with a workspace");
    if ((o.coarse_op != EECMG_COARSE_GALERKIN_RMS && o.coarse_op != EECMG_COARSE_GALERKIN_RENORM) ||
        (o.stop != EECMG_STOP_FIXED && o.stop != EECMG_STOP_DISCREPANCY) || !(o.c > 1.0) ||
        !(o.delta >= 0.0) || o.diffusion_steps < 0 || o.diffusion_steps > 64 || !(o.conv_tol >= 0.0) ||
        !std::isfinite(o.s_scale))
        return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_plan: invalid option");
    const int nk = psf_w * psf_h * psf_d;
    std::vector<double> K(psf, psf + nk);
    double ksum = 0.0;
    for (double v : K) {
        if (!std::isfinite(v)) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_plan: PSF not finite");
        ksum += v;
    }
    if (!(ksum > 0.0)) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_plan: PSF sum must be positive");
    for (int i = 0; i < nk; ++i)  // MR-II needs H symmetric: K(d) = K(-d)
        if (std::fabs(K[i] - K[nk - 1 - i]) > 1e-12 * std::fabs(ksum))
            return set_error(EECMG_ERR_UNSUPPORTED, "eecmg_vol_plan: MR-II needs a centrosymmetric PSF");
    if (iters)
        for (int l = 0; l < levels; ++l)
            if (iters[l] < 0) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_plan: iters < 0");

    auto* P = new eecmg_vol_s();
    P->W = width;
    P->H = height;
    P->D = depth;
    P->L = levels;
    P->tau = alpha;
    P->kpm = k;
    P->opt = o;
    const int L = levels;
    P->ds.resize(L);
    P->hs.resize(L);
    P->ws.resize(L);
    P->m.resize(L);
    P->ds[L - 1] = depth;
    P->hs[L - 1] = height;
    P->ws[L - 1] = width;
    for (int l = L - 1; l > 0; --l) {
        P->ds[l - 1] = (P->ds[l] + 1) / 2;
        P->hs[l - 1] = (P->hs[l] + 1) / 2;
        P->ws[l - 1] = (P->ws[l] + 1) / 2;
    }
    for (int l = 0; l < L; ++l) P->m[l] = iters ? iters[l] : schedule_m(L, l + 1);
    P->n.resize(L);
    P->n4.resize(L);
    for (int l = 0; l < L; ++l) {
        P->n[l] = (long long)P->ds[l] * P->hs[l] * P->ws[l];
        P->n4[l] = (P->n[l] + 3) / 4;
    }
    // level PSFs (Eq. 14 in 3-D; RENORM rescales to the fine PSF's sum)
    std::vector<std::vector<double>> Kl(L);
    std::vector<int> kdl(L), khl(L), kwl(L);
    Kl[L - 1] = K;
    kdl[L - 1] = psf_d;
    khl[L - 1] = psf_h;
    kwl[L - 1] = psf_w;
    for (int l = L - 1; l > 0; --l) {
        const double rho = (double)P->n[l] / (double)P->n[l - 1];
        const int rz = kdl[l] / 2, ry = khl[l] / 2, rx = kwl[l] / 2;
        const int cz = rz / 2, cy = ry / 2, cx = rx / 2;
        kdl[l - 1] = 2 * cz + 1;
        khl[l - 1] = 2 * cy + 1;
        kwl[l - 1] = 2 * cx + 1;
        Kl[l - 1].assign((size_t)kdl[l - 1] * khl[l - 1] * kwl[l - 1], 0.0);
        for (int a = -cz; a <= cz; ++a)
            for (int b = -cy; b <= cy; ++b)
                for (int c = -cx; c <= cx; ++c)
                    Kl[l - 1][((size_t)(a + cz) * khl[l - 1] + (b + cy)) * kwl[l - 1] + (c + cx)] =
                        rho * Kl[l][((size_t)(2 * a + rz) * khl[l] + (2 * b + ry)) * kwl[l] + (2 * c + rx)];
        if (o.coarse_op == EECMG_COARSE_GALERKIN_RENORM) {
            double s = 0.0;
            bool nz = false;
            for (double v : Kl[l - 1]) {
                s += v;
                nz = nz || v != 0.0;
            }
            if (s != 0.0 && nz)
                for (double& v : Kl[l - 1]) v *= ksum / s;
        }
    }
    P->taps.resize(L);
    P->tapsT.resize(L);
    P->gt.resize(L);
    P->gtT.resize(L);
    size_t ntaps = 0;
    for (int l = 0; l < L; ++l) {
        make_vol_taps(Kl[l], kdl[l], khl[l], kwl[l], false, &P->taps[l], &P->gt[l]);
        make_vol_taps(Kl[l], kdl[l], khl[l], kwl[l], true, &P->tapsT[l], &P->gtT[l]);
        ntaps += P->gt[l].size() + P->gtT[l].size() + 2;
    }
    // workspace: g and u per level, 8 solver vectors, taps, barriers, partials
    eecmg_status st = EECMG_OK;
    cudaError_t e = cudaGetDevice(&P->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&P->sms, cudaDevAttrMultiProcessorCount, P->device);
    if (e != cudaSuccess) {
        delete P;
        return set_error(EECMG_ERR_CUDA, std::string("eecmg_vol_plan: ") + cudaGetErrorString(e));
    }
    // few slices per block to march (two blocks per SM): tiles (62 x 146 x 25, r = 3, 1.2 slices
    // a block: solve 121 us marched, 83 us in tiles; 256^3, 34 slices a block: 46 against 113 us
    // a convolution).  SmallTile has both sides around the line.
    for (int l = 0; l < L; ++l)
        for (VolTaps* t : {&P->taps[l], &P->tapsT[l]})
            if (t->form == VF_SEP && level_units(P->ds[l], P->hs[l], P->ws[l], *t) < 2LL * t->r * 2 * P->sms)
                t->form = VF_SMALL;
    P->grid.resize(L);
    int maxgrid = 1;
    for (int l = 0; l < L; ++l) {
        // the attribute belongs to the kernel, which plans of every form share
        const int r = P->taps[l].r;
        size_t most = 0;
        for (int f : {VF_SEP, VF_DENSE, VF_SPARSE, VF_SMALL}) most = std::max(most, form_bytes(r, f));
        const size_t smem = form_bytes(r, P->taps[l].form);
        e = cudaFuncSetAttribute(vol_kernels().solve[r], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)most);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(vol_kernels().apply[r], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)most);
        int per = 0;
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, vol_kernels().solve[r], NTHREADS, smem);
        if (e != cudaSuccess || per < 1) {
            delete P;
            return set_error(EECMG_ERR_CUDA, "eecmg_vol_plan: level solve does not fit an SM");
        }
        const long long want =
            std::max<long long>(level_units(P->ds[l], P->hs[l], P->ws[l], P->taps[l]), (P->n4[l] + NTHREADS - 1) / NTHREADS);
        const long long cap = (long long)per * P->sms;
        P->grid[l] = (int)std::max<long long>(1, std::min(want, cap));
        maxgrid = std::max(maxgrid, P->grid[l]);
    }
    size_t off = 0;
    std::vector<size_t> goff(L), uoff(L), voff(8);
    for (int l = 0; l < L; ++l) {
        goff[l] = off;
        off = align256(off + (size_t)P->n4[l] * 16);
        uoff[l] = off;
        off = align256(off + (size_t)P->n4[l] * 16);
    }
    for (int i = 0; i < 8; ++i) {
        voff[i] = off;
        off = align256(off + (size_t)P->n4[L - 1] * 16);
    }
    const size_t taps_off = off;
    off = align256(off + ntaps * sizeof(int4));
    const size_t gs_off = off;
    off = align256(off + (size_t)L * sizeof(GroupSync));
    const size_t out_off = off;
    off = align256(off + (size_t)L * 4 * sizeof(double));
    const size_t part_off = off;
    off = align256(off + (size_t)2 * maxgrid * NPART * sizeof(double));
    e = cudaMalloc((void**)&P->wsp, off);
    if (e != cudaSuccess) {
        cudaGetLastError();
        delete P;
        return set_error(EECMG_ERR_OOM, "eecmg_vol_plan: workspace allocation failed");
    }
    P->ws_bytes = off;
    e = cudaMemset(P->wsp, 0, off);
    P->g.resize(L);
    P->u.resize(L);
    for (int l = 0; l < L; ++l) {
        P->g[l] = (float*)(P->wsp + goff[l]);
        P->u[l] = (float*)(P->wsp + uoff[l]);
    }
    for (int i = 0; i < 8; ++i) P->vec[i] = (float*)(P->wsp + voff[i]);
    P->dtaps = (int4*)(P->wsp + taps_off);
    P->gs = (GroupSync*)(P->wsp + gs_off);
    P->out = (double*)(P->wsp + out_off);
    P->partials = (double*)(P->wsp + part_off);
    std::vector<int4> all;
    P->dtap_off.resize(2 * L);
    for (int l = 0; l < L; ++l) {
        P->dtap_off[2 * l] = all.size();
        all.insert(all.end(), P->gt[l].begin(), P->gt[l].end());
        all.push_back(make_int4(0, 0, 0, 0));
        P->dtap_off[2 * l + 1] = all.size();
        all.insert(all.end(), P->gtT[l].begin(), P->gtT[l].end());
        all.push_back(make_int4(0, 0, 0, 0));
    }
    if (e == cudaSuccess)
        e = cudaMemcpy(P->dtaps, all.data(), all.size() * sizeof(int4), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&P->cap, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
        st = set_error(EECMG_ERR_CUDA, std::string("eecmg_vol_plan: ") + cudaGetErrorString(e));
        cudaFree(P->wsp);
        delete P;
        return st;
    }
    *out = P;
    return EECMG_OK;
}

eecmg_status eecmg_vol_plan_destroy(eecmg_vol_t P) {
    if (!P) return EECMG_OK;
    cudaDeviceSynchronize();
    if (P->gexec) cudaGraphExecDestroy(P->gexec);
    if (P->cap) cudaStreamDestroy(P->cap);
    for (cudaEvent_t e : P->ev) cudaEventDestroy(e);
    if (P->wsp) cudaFree(P->wsp);
    delete P;
    return EECMG_OK;
}

eecmg_status eecmg_vol_plan_info(eecmg_vol_t P, int* levels, int* level_w, int* level_h,
                                 int* level_d, int* iters, size_t* workspace_bytes) {
    if (!P) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_plan_info: NULL plan");
    if (levels) *levels = P->L;
    for (int l = 0; l < P->L; ++l) {
        if (level_w) level_w[l] = P->ws[l];
        if (level_h) level_h[l] = P->hs[l];
        if (level_d) level_d[l] = P->ds[l];
        if (iters) iters[l] = P->m[l];
    }
    if (workspace_bytes) *workspace_bytes = P->ws_bytes;
    return EECMG_OK;
}

eecmg_status eecmg_vol_restore(eecmg_vol_t P, const float* g, float* u, cudaStream_t s) {
    if (!P || !g || !u) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_restore: NULL argument");
    const size_t bytes = (size_t)P->n[P->L - 1] * sizeof(float);
    VCK(cudaMemcpyAsync(P->g[P->L - 1], g, bytes, cudaMemcpyDeviceToDevice, s));
    eecmg_status st = run_cascade(P, s);
    if (st != EECMG_OK) return st;
    VCK(cudaMemcpyAsync(u, P->u[P->L - 1], bytes, cudaMemcpyDeviceToDevice, s));
    return EECMG_OK;
}

eecmg_status eecmg_vol_restore_host(eecmg_vol_t P, const float* g_host, float* u_host,
                                    cudaStream_t s) {
    if (!P || !g_host || !u_host)
        return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_restore_host: NULL argument");
    const size_t bytes = (size_t)P->n[P->L - 1] * sizeof(float);
    VCK(cudaMemcpyAsync(P->g[P->L - 1], g_host, bytes, cudaMemcpyHostToDevice, s));
    eecmg_status st = run_cascade(P, s);
    if (st != EECMG_OK) return st;
    VCK(cudaMemcpyAsync(u_host, P->u[P->L - 1], bytes, cudaMemcpyDeviceToHost, s));
    VCK(cudaStreamSynchronize(s));
    return EECMG_OK;
}

eecmg_status eecmg_vol_plan_stats(eecmg_vol_t P, int* iters_done, double* res_rms) {
    if (!P) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_plan_stats: NULL plan");
    VCK(cudaDeviceSynchronize());
    std::vector<double> h(4 * (size_t)P->L);
    VCK(cudaMemcpy(h.data(), P->out, h.size() * sizeof(double), cudaMemcpyDeviceToHost));
    std::vector<GroupSync> gs(P->L);
    VCK(cudaMemcpy(gs.data(), P->gs, gs.size() * sizeof(GroupSync), cudaMemcpyDeviceToHost));
    for (int l = 0; l < P->L; ++l) {
        if (iters_done) iters_done[l] = (int)h[4 * l];
        if (res_rms) res_rms[l] = std::sqrt(h[4 * l + 1] / (double)P->n[l]);
        if (gs[l].err) return set_error(EECMG_ERR_TIMEOUT, "eecmg_vol_plan_stats: a grid barrier timed out");
    }
    return EECMG_OK;
}

eecmg_status eecmg_vol_apply_H(eecmg_vol_t P, int level, const float* x, float* y, int transpose,
                               cudaStream_t s) {
    eecmg_status st = check_level(P, level, "eecmg_vol_apply_H");
    if (st != EECMG_OK) return st;
    if (!x || !y || x == y) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_apply_H: bad buffers");
    return launch_apply(P, level, transpose != 0, x, y, s);
}

eecmg_status eecmg_vol_start_level(eecmg_vol_t P, int level, const float* u1, const float* u2,
                                   float* out, cudaStream_t s) {
    eecmg_status st = check_level(P, level, "eecmg_vol_start_level");
    if (st != EECMG_OK) return st;
    if (level < 2 || !u1 || !u2 || !out)
        return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_start_level: needs level >= 2 and buffers");
    return launch_start(P, level, u1, u2, out, s);
}

eecmg_status eecmg_vol_smooth(eecmg_vol_t P, int level, const float* x, float* y, cudaStream_t s) {
    eecmg_status st = check_level(P, level, "eecmg_vol_smooth");
    if (st != EECMG_OK) return st;
    if (!x || !y || x == y) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_smooth: bad buffers");
    VCK(launch_vol_smooth(x, P->ds[level], P->hs[level], P->ws[level], (float)P->opt.s_scale, y, s));
    return EECMG_OK;
}

eecmg_status eecmg_vol_denoise(eecmg_vol_t P, int level, const float* x, float* y, cudaStream_t s) {
    eecmg_status st = check_level(P, level, "eecmg_vol_denoise");
    if (st != EECMG_OK) return st;
    if (!x || !y || x == y) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_denoise: bad buffers");
    const int d = P->ds[level], h = P->hs[level], w = P->ws[level];
    VCK(launch_vol_denoise(x, d, h, w, (float)(1.0 / (P->kpm * P->kpm)), (float)P->tau, P->vec[7], y, s));
    return EECMG_OK;
}

eecmg_status eecmg_vol_restrict(eecmg_vol_t P, int level, const float* fine, float* coarse,
                                cudaStream_t s) {
    eecmg_status st = check_level(P, level, "eecmg_vol_restrict");
    if (st != EECMG_OK) return st;
    if (level >= P->L - 1 || !fine || !coarse)
        return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_restrict: level must be below the finest");
    k_vol_restrict<<<vgrid(P->ds[level], P->hs[level], P->ws[level]), VTHREADS, 0, s>>>(fine, P->hs[level + 1], P->ws[level + 1],
                                                          coarse, P->ds[level], P->hs[level],
                                                          P->ws[level]);
    VCK(cudaGetLastError());
    return EECMG_OK;
}

eecmg_status eecmg_vol_level_solve(eecmg_vol_t P, int level, const float* g, float* u, int m,
                                   cudaStream_t s) {
    eecmg_status st = check_level(P, level, "eecmg_vol_level_solve");
    if (st != EECMG_OK) return st;
    if (!g || !u || m < 0) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_level_solve: bad arguments");
    const size_t bytes = (size_t)P->n[level] * sizeof(float);
    VCK(cudaMemcpyAsync(P->g[level], g, bytes, cudaMemcpyDeviceToDevice, s));
    VCK(cudaMemcpyAsync(P->u[level], u, bytes, cudaMemcpyDeviceToDevice, s));
    const int keep = P->m[level];
    P->m[level] = m;
    st = launch_solve(P, level, false, s);
    P->m[level] = keep;
    if (st != EECMG_OK) return st;
    VCK(cudaMemcpyAsync(u, P->u[level], bytes, cudaMemcpyDeviceToDevice, s));
    return EECMG_OK;
}

eecmg_status eecmg_vol_plan_profile(eecmg_vol_t P, int enable) {
    if (!P) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_plan_profile: NULL plan");
    if (enable && P->ev.empty()) {
        P->ev.resize(4 * (size_t)P->L);
        for (auto& e : P->ev) VCK(cudaEventCreate(&e));
    }
    P->ev_used.assign(4 * (size_t)P->L, 0);
    P->prof = enable != 0;
    return EECMG_OK;
}

eecmg_status eecmg_vol_plan_profile_read(eecmg_vol_t P, double* start_ms, double* solve_ms,
                                         double* solve_bytes_out) {
    if (!P || !P->prof) return set_error(EECMG_ERR_INVALID_ARG, "eecmg_vol_plan_profile_read: profiling is off");
    VCK(cudaDeviceSynchronize());
    std::vector<double> h(4 * (size_t)P->L);
    VCK(cudaMemcpy(h.data(), P->out, h.size() * sizeof(double), cudaMemcpyDeviceToHost));
    for (int l = 0; l < P->L; ++l) {
        float a = 0.f, b = 0.f;
        if (P->ev_used[4 * l] && P->ev_used[4 * l + 1])
            VCK(cudaEventElapsedTime(&a, P->ev[4 * l], P->ev[4 * l + 1]));
        if (P->ev_used[4 * l + 2] && P->ev_used[4 * l + 3])
            VCK(cudaEventElapsedTime(&b, P->ev[4 * l + 2], P->ev[4 * l + 3]));
        if (start_ms) start_ms[l] = a;
        if (solve_ms) solve_ms[l] = b;
        if (solve_bytes_out) solve_bytes_out[l] = solve_bytes(P, l, (int)h[4 * l], (int)h[4 * l + 2]);
    }
    return EECMG_OK;
}

}  // extern "C"
