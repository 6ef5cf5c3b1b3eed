// complex64 FFT passes for any two-stage plan (fft_lines.cu).
#pragma once
#include "pw_internal.cuh"

namespace pw {
namespace fl {

// Whether the passes cover the box: every length with a two-stage plan, up to 256.
bool covers(const FftPlan& plan);

// Pass 1 (sphere -> half-box planes), pass 2 (x-lines) and pass 3 (planes -> sphere, + kinetic term
// or with rec the recurrence) of launch_local_apply<float> for nb bands, on the same layouts.
cudaError_t inverse_planes(const FftPlan& plan, const float2* tw, const SphereDev& sp, const float2* psi,
                           int64_t ldpsi, float2* hb, int64_t hb_bs, int nb, cudaStream_t st);
cudaError_t xlines(const FftPlan& plan, const float2* tw, const SphereDev& sp, const float* vperm, float2* hb,
                   int64_t hb_bs, int nb, cudaStream_t st);
cudaError_t forward_planes(const FftPlan& plan, const float2* tw, const SphereDev& sp, const float* kin, float2* hb,
                           int64_t hb_bs, const float2* psi, int64_t ldpsi, float2* out, int64_t ldout, int nb,
                           cudaStream_t st, const Pass3Rec* rec);

}  // namespace fl
}  // namespace pw
