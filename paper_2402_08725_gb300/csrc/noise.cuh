// The transform form of the noise propagation's correlation (noise_fft.cu), internal.
#pragma once

#include "common.cuh"

namespace sr {

// L = R1 R2: transform size, n x n output tiles of T x T per realisation.
struct NoiseFft {
    int L = 0, R1 = 0, n = 0, T = 0;
};
constexpr int kNoiseMaxL = 160;  // the largest transform
// The kernel spectrum S [L][L] (scaled by 1 / L^2), the twiddles tw [L], and the tap offset sh: tap
// q of s_1 acts at (q - sh) mod L.  gain[k]: what a transform there and back multiplies frequency k of
// one axis by, for its roots of unity are rounded (noise_fft_gain); S is divided by it.  L = 0: none.
struct NoiseSpec {
    float2 *S = nullptr, *tw = nullptr;
    int L = 0, R1 = 1, sh = 0;
    double gain[kNoiseMaxL];
};
// gain[k], k < L, of the plan's transforms.
void noise_fft_gain(const NoiseFft &plan, double *gain);
// The cheapest plan (n^2 L^2) whose transforms fit smem_optin bytes of shared memory; false if none.
bool noise_fft_plan(int F, int K, int smem_optin, NoiseFft *plan);
// Configures the transform kernel on the current device; *resident = its blocks per SM.
sr_status noise_fft_prepare(const NoiseFft &plan, int *resident);
// y[b] = S_1^T x[b] for the B realisations of a batch; nothing where *skip (on the device) is set.
sr_status launch_noise_fft(const NoiseFft &plan, const float *x, const float2 *S, const float2 *tw, int F, int K, int B,
                           int n_sms, const int *skip, float *y, cudaStream_t st);

}  // namespace sr
