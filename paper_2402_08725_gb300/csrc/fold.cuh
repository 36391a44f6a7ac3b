// The D-folded narrow-PSF kernels (internal; shared by the per-problem and the batched set-up).
#pragma once

#include "ffsum.cuh"

namespace sr {

// kappa_{i,phi}(tau) for tau in [tau_lo, tau_lo + Tk)^2, element idx of [f*f][Tk][Tk] of one epoch
// (phi = phy*f + phx): kappa(t) = sum_{a,b<f} s[t + (a,b) + o] with t = f*tau - phi, o = K/2, the
// sum over the f x f block of D taken as a compensated FP32 pair (48 bits) in a fixed order and rounded
// once: in FP64, which runs at 2 operations a clock per SM, the folding of 2000 PSFs of 64 x 64 was bound
// by that pipe (with 64-bit indexes too; 32 renewed fields 1001 -> 967 us an evaluation).
__device__ __forceinline__ float kappa_fold(const float *__restrict__ si, int K, int f, int Tk, int tau_lo,
                                            int idx) {
    const int ph = idx / (Tk * Tk), r = idx - ph * Tk * Tk;  // at most 64 x 512^2 elements: 32 bits
    const int ty = r / Tk, tx = r - ty * Tk;
    const int phy = ph / f, phx = ph - phy * f, o = K / 2;
    const int t_y = f * (tau_lo + ty) - phy;
    const int t_x = f * (tau_lo + tx) - phx;
    FSum acc = fsum_zero();
    for (int a = 0; a < f; ++a) {
        const int qy = t_y + a + o;
        if (qy < 0 || qy >= K) continue;
        for (int b = 0; b < f; ++b) {
            const int qx = t_x + b + o;
            if (qx < 0 || qx >= K) continue;
            acc = fsum_add(acc, si[qy * K + qx]);
        }
    }
    return acc.hi + acc.lo;
}

}  // namespace sr
