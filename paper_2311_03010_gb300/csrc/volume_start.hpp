// volume_start.hpp -- launchers of the operators that start a level of the
// volume cascade (volume_start.cu): dense d x h x w FP32 volumes, asynchronous
// on the stream, in != out.
#pragma once

#include <cuda_runtime.h>

namespace eecmg {
namespace vol {

// Pi on the level-(l-1) grid (d1 x h1 x w1) from u1 and the level-(l-2) solution u2.
cudaError_t launch_vol_pi(const float* u1, int d1, int h1, int w1, const float* u2, int d2, int h2, int w2,
                          float* out, cudaStream_t s);
// P: the three-point quadratic rule from d1 x h1 x w1 onto d x h x w.
cudaError_t launch_vol_quad(const float* ut, int d1, int h1, int w1, float* out, int d, int h, int w,
                            cudaStream_t s);
cudaError_t launch_vol_smooth(const float* u, int d, int h, int w, float scale, float* out, cudaStream_t s);
// One Perona-Malik step; c: a d x h x w buffer for the diffusivities.
cudaError_t launch_vol_denoise(const float* u, int d, int h, int w, float ik2, float tau, float* c, float* out,
                               cudaStream_t s);

}  // namespace vol
}  // namespace eecmg
