// Frequency-domain form of the deconvolution loss and gradient: in-place transforms of real
// image pairs (sm_103a).
//
// The D-folded polyphase model is a sum over phases phi of data-grid convolutions,
// M_i = sum_phi kappa_{i,phi} * F_phi (Eq. 8-10 with the block sum folded into the kernels), and
// its adjoint a correlation per phase.  With circular transforms of size L x L,
// L >= N + max(tau_hi, -tau_lo), the wrap-around never reaches the N x N output, so
//     M_i = IDFT( sum_phi Khat_{i,phi} (Hhat_phi + Phat_{i,phi}) )          on [0,N)^2,
//     dL/dh_phi = IDFT( sum_i conj(Khat_{i,phi}) ehat_i )                   on [0,N)^2,
// exactly up to rounding.  Khat (spectra of the folded kernels) are computed at set_psfs, Hhat
// (the phase images of h) once per evaluation, the point sources' spectra are outer products of
// 1-D DFTs of the sampled Gaussian window, and their gradients come from Parseval's identity.
//
// Every transform is a complex L x L transform of two epochs at once (real and imaginary parts), in
// one buffer in shared memory.  A length-L transform, L = R1 R2, is two passes of in-register DFTs
// that read and write the same positions:
//   pass A: for each n2 < R2, the R1-point DFT over n1 of x[n2 + R2 n1], times W_L^(n2 k1),
//           written back to positions n2 + R2 k1;
//   pass B: for each k1 < R1, the R2-point DFT of the R2 consecutive values at R2 k1 + n2,
//           written back in place: X[k1 + R1 k2] lands at position R2 k1 + k2.
// Spectra therefore live in "digit-transposed" order (frequency k at position R2 (k mod R1) + k / R1);
// the inverse runs the passes backwards (B then A) and returns the natural spatial order.
//
// The chunk kernel's limits are the loads of the spectral passes (two thirds of its time: the kernel
// spectra come from DRAM once and half of their second reading too, with 152 blocks' working sets
// beyond the L2) and the latency of its passes at 16 warps per SM.  So
//   * the spectral products are fused with the outermost column passes: a thread owns the R2 rows
//     ky = k1 + R1 k2 of one column kx, so the model spectrum goes from registers into the inverse
//     pass B, and the residual spectrum from the forward pass B into the adjoint products;
//   * the residual is formed between the inverse and the forward row pass A in registers;
//   * two epochs travel side by side through the spectral arithmetic and pass B along y (C2 of
//     cpack.cuh, the kernel spectra stored as (re_a, re_b, im_a, im_b)), one packed instruction for
//     both.  Column kx and its mirror -kx are separated or joined before pass B, where the relation
//     is the same: with a, b the two epochs' values after the DFT over k2 and the twiddle,
//     Z(kx) = a + i b and Z(-kx) = conj(a) + i conj(b) at the mirrored residue (R1 - k1) mod R1.
// That leaves six round trips through shared memory and nine barriers per pair, and 0.4 of the
// instructions of ten passes over the buffer with scalar arithmetic.  Against that version, with the
// same 16 warps (transform kernels, us): 8 fields of 304 epochs at L = 144 866 -> 648, L = 128 788 -> 522,
// L = 112 545 -> 443 (four sources, 4 fields: 552 -> 332); 16 fields at L = 80 568 -> 433, L = 64
// 394 -> 294, L = 48 262 -> 197; 2 fields of 300 epochs with four sources at L = 80 172 -> 128.
// Rows are R1x groups of R2x = 16 (or 8) positions padded to 17 (9): a row pitch of R1x mod 16 keeps
// both row passes free of bank conflicts; along y R1y = 16 (8), so pass B has the few points that
// fit in registers beside the spectra.
#include <math.h>

#include <algorithm>
#include <functional>
#include <queue>
#include <vector>

#include "common.cuh"
#include "cplx.cuh"
#include "ffsum.cuh"
#include "fft_pair.cuh"
#include "kernels.cuh"

namespace sr {
namespace {

// --- the per-epoch chunk kernel ---------------------------------------------------------------
constexpr int kChunkThreads = 512;

struct PrShared {
    // the work item's parameters: amplitudes a_{i,k}, epoch shifts delta_i, backgrounds gamma_i of
    // its epochs, and the source positions c_k (loaded once per item)
    float ia[kFftChunk * kFftMaxSources];
    float id[2 * kFftChunk];
    float ig[kFftChunk];
    float ic[2 * kFftMaxSources];
    float2 cs[2][2][kChunkThreads / 32];  // chi^2 | sum e of both epochs of the warp's pair, per warp
    // per-warp Parseval sums [epoch][source][a | x | y]: four pairs of one source, or one of four
    float red[8 * 3][kChunkThreads / 32];
    int item;
};
__shared__ PrShared pr_sh;

template <int L>
struct Ck {
    static constexpr int R2X = L % 16 == 0 ? 16 : 8, R1X = L / R2X, SX = R2X + 1;
    static constexpr int R1Y = R2X, R2Y = L / R1Y;
    static constexpr int P = R1X * SX;             // row pitch (float2)
    static constexpr int ZN = (L * P + 1) & ~1;    // float2 per pair buffer
    static constexpr int H = L / 2 + 1, HP = H + 1;
    static_assert(R1X * R2X == L && R1Y * R2Y == L && L % 4 == 0, "transform size not in the list");
};
// physical column of frequency kx
template <int L>
__device__ __forceinline__ int ckcol(int kx) {
    return (kx % Ck<L>::R1X) * Ck<L>::SX + kx / Ck<L>::R1X;
}

// shared memory of GP pair buffers, the window-profile tables and the roots of unity
template <int L>
__host__ __device__ constexpr int ck_smem(int GP, int M, int f) {
    return (GP * Ck<L>::ZN + 2 * GP * M * f * 4 * Ck<L>::H + L) * 8;
}
constexpr int kChunkSmem = 229500;  // the opt-in limit (about 227 KB) less the static part
// epoch pairs per group for at most one source: 4 or 2 where they fit (at f = 2), else 1
template <int L>
__host__ __device__ constexpr int pr_gpmax() {
    return ck_smem<L>(4, 1, 2) <= kChunkSmem ? 4 : ck_smem<L>(2, 1, 2) <= kChunkSmem ? 2 : 1;
}

// profile tables: [pair of the group][source][phase][kind][H] of (re_a, re_b, im_a, im_b); kind 0 gx,
// 1 d gx, 2 gy, 3 d gy
__device__ __forceinline__ int prof_at(int g, int k, int ph, int kind, int M, int f, int H) {
    return (((g * M + k) * f + ph) * 4 + kind) * H;
}

// 1-D DFTs (frequencies 0 .. L/2) of the window profiles g1(u - c) and g1(u - c) (u - c) / sigma^2 on
// each phase's sub-grid u = f m + phase, for the epochs of np pairs (zero for a missing last one).
// The samples first (into scratch), then each frequency's sum over them.
template <int L>
__device__ __forceinline__ void window_profiles(const FieldDev &fd, const PrShared &sh, int e_item, int ne, int np,
                                                float2 *scratch, float4 *prof, const float2 *W) {
    constexpr int H = Ck<L>::H;
    const int f = fd.f, F = fd.F, M = fd.M, tid = threadIdx.x, nt = blockDim.x;
    const float u0 = 0.5f * (float)(F - 1);
    const int taps = (kWin + f - 1) / f;
    // first sub-grid position at or after the window's first pixel
    auto first = [&](int e, int k, int xy, int phs) {
        const float cc = u0 + (float)f * (sh.ic[2 * k + xy] + sh.id[2 * (e_item + e) + xy]);
        const int lo = (int)floorf(cc) - kWinLo, d = lo - phs;
        return d >= 0 ? (d + f - 1) / f : -((-d) / f);
    };
    const int n_s = ne * M * f * 2 * taps;
    for (int idx = tid; idx < n_s; idx += nt) {
        const int q = idx / taps, tap = idx - q * taps;
        const int xy = q & 1, kf = (q >> 1) % (M * f), e = (q >> 1) / (M * f);
        const int k = kf / f, phs = kf - k * f;
        const float cpos = sh.ic[2 * k + xy], dl = sh.id[2 * (e_item + e) + xy];
        const int lo = (int)floorf(u0 + (float)f * (cpos + dl)) - kWinLo;
        const int u = f * (first(e, k, xy, phs) + tap) + phs;
        float2 g = make_float2(0.f, 0.f);
        if (u >= 0 && u < F && u < lo + kWin) {
            const float t = src_offset(u, F, f, cpos, dl);
            g.x = kGauss1Norm * exp2f(-t * t);
            g.y = g.x * t * kGaussInvSig2;
        }
        scratch[idx] = g;
    }
    __syncthreads();
    float *out = reinterpret_cast<float *>(prof);
    const int n_e = 2 * np * M * f * 2 * H;
    for (int idx = tid; idx < n_e; idx += nt) {
        const int q = idx / H, kk = idx - q * H;
        const int xy = q & 1, kf = (q >> 1) % (M * f), e = (q >> 1) / (M * f);
        const int k = kf / f, phs = kf - k * f;
        float2 v = make_float2(0.f, 0.f), vd = make_float2(0.f, 0.f);
        if (e < ne) {
            const int m0 = first(e, k, xy, phs) % L;
            int j = (kk * (m0 < 0 ? m0 + L : m0)) % L;
            const float2 *sg = scratch + q * taps;
            for (int t = 0; t < taps; ++t) {
                const float2 g = sg[t], w = W[j];
                v.x += g.x * w.x;
                v.y += g.x * w.y;
                vd.x += g.y * w.x;
                vd.y += g.y * w.y;
                j += kk;
                if (j >= L) j -= L;
            }
        }
        float *o = out + 4 * (prof_at(e >> 1, k, phs, 2 * xy, M, f, H) + kk) + (e & 1);
        o[0] = v.x;
        o[2] = v.y;
        o[4 * H] = vd.x;
        o[4 * H + 2] = vd.y;
    }
}

// Row k2 of a unit (ky = k1 + R1Y k2) in the profile tables, which hold ky <= L/2: the position, and
// the sign of the imaginary part.  Both halves of the rows are known at compile time; only the middle
// row of an odd R2Y depends on k1.
template <int L>
__device__ __forceinline__ int prof_row(int k1, int k2) {
    using G = Ck<L>;
    const int ky = k1 + G::R1Y * k2;
    if (2 * k2 + 1 < G::R2Y) return ky;
    if (2 * k2 + 1 > G::R2Y) return L - ky;
    return min(ky, L - ky);
}
// y with the sign applied where it depends on k1
template <int L>
__device__ __forceinline__ float4 prof_val(const float4 *y, int k1, int k2) {
    float4 v = y[prof_row<L>(k1, k2)];
    if (2 * k2 + 1 == Ck<L>::R2Y && 2 * (k1 + Ck<L>::R1Y * k2) > L) {
        v.z = -v.z;
        v.w = -v.w;
    }
    return v;
}
template <int L>
__host__ __device__ constexpr bool prof_conj(int k2) {  // the row's values are the conjugates of the table's
    return 2 * k2 + 1 > Ck<L>::R2Y;
}

// Model spectra sum_phi Khat_{e,phi} (Hhat_phi + sum_k a_{e,k} gx gy) of the group's epochs and the
// inverse pass B along y.  A unit is column kx and residue k1 of one pair: rows ky = k1 + R1Y k2.
// Bound by the latency of the spectra's loads (16 warps per SM), so all rows of a phase are loaded
// before any is used: 9 rows of 24 bytes per thread in flight at L = 144.  (In an earlier form of this
// pass, 8 fields of 304 epochs at L = 144: the whole phase 805 us, half of it 941, two rows kept ahead of
// their use 1039, for loads of several ages wait for one another on a warp's six scoreboards.  Nor may
// it spill much: beside 177 KB of buffers the L1 is about 28 KB.  44 bytes are left at L = 72 and 144, 24 at
// L = 128, for one source; 44-84 at L = 56, 72, 112, 128 and 144, 16 at L = 96, for up to four.)
// prof_off, w_off: the profile tables and the roots of unity in pr_dyn (float2).
template <int L, int MS>
__device__ __noinline__ void spec_model(const FieldDev &fd, const float2 *__restrict__ hh, const float4 *__restrict__ kh,
                                        int a0, int ne, int prof_off, int w_off) {
    using G = Ck<L>;
    constexpr int H = G::H, HP = G::HP, LHP = L * HP, ZN = G::ZN, P = G::P, R1Y = G::R1Y, R2Y = G::R2Y;
    constexpr int UNITS = H * R1Y;
    const int f = fd.f, M = fd.M, nph = f * f, np = (ne + 1) / 2;
    const float4 *prof0 = reinterpret_cast<const float4 *>(pr_dyn + prof_off);
    const float2 *W = pr_dyn + w_off;
    const unsigned long long pol = l2_policy_last();
    for (int t = threadIdx.x; t < np * UNITS; t += blockDim.x) {
        const int g = t / UNITS, r = t - g * UNITS;
        const int k1 = r / H, kx = r - k1 * H;
        const float2 *hp = hh + k1 * HP + kx;
        const float4 *kp = kh + (long long)g * nph * LHP + k1 * HP + kx;
        C2 m[R2Y];
#pragma unroll
        for (int k2 = 0; k2 < R2Y; ++k2) m[k2].re = m[k2].im = make_float2(0.f, 0.f);
        int phy = 0, phx = 0;
        for (int ph = 0; ph < nph; ++ph) {
            float2 hv[R2Y];
            float4 kv[R2Y];
#pragma unroll
            for (int k2 = 0; k2 < R2Y; ++k2) {
                hv[k2] = ldg_hint(hp + ph * LHP + k2 * R1Y * HP, pol);
                kv[k2] = ldg_hint(kp + ph * LHP + k2 * R1Y * HP, pol);
            }
            // a_k gx of the column, both epochs
            C2 src[MS];
            const float4 *yt = prof0 + prof_at(g, 0, phy, 2, M, f, H);
#pragma unroll
            for (int k = 0; k < MS; ++k) {
                src[k].re = src[k].im = make_float2(0.f, 0.f);
                if (k < M) {
                    const float4 x = prof0[prof_at(g, k, phx, 0, M, f, H) + kx];
                    const float2 a = make_float2(pr_sh.ia[(a0 + 2 * g) * M + k],
                                                 2 * g + 1 < ne ? pr_sh.ia[(a0 + 2 * g + 1) * M + k] : 0.f);
                    src[k].re = f2mul(a, make_float2(x.x, x.y));
                    src[k].im = f2mul(a, make_float2(x.z, x.w));
                }
            }
#pragma unroll
            for (int k2 = 0; k2 < R2Y; ++k2) {
                float2 sre = f2dup(hv[k2].x), sim = f2dup(hv[k2].y);
#pragma unroll
                for (int k = 0; k < MS; ++k) {
                    if (k < M) {
                        const float4 y = prof_val<L>(yt + k * f * 4 * H, k1, k2);
                        const float2 yre = make_float2(y.x, y.y), yim = make_float2(y.z, y.w);
                        sre = f2fma(src[k].re, yre, sre);
                        sim = f2fma(src[k].im, yre, sim);
                        if (prof_conj<L>(k2)) {
                            sre = f2fma(src[k].im, yim, sre);
                            sim = f2nfma(src[k].re, yim, sim);
                        } else {
                            sre = f2nfma(src[k].im, yim, sre);
                            sim = f2fma(src[k].re, yim, sim);
                        }
                    }
                }
                const float2 kre = make_float2(kv[k2].x, kv[k2].y), kim = make_float2(kv[k2].z, kv[k2].w);
                m[k2].re = f2nfma(kim, sim, f2fma(kre, sre, m[k2].re));
                m[k2].im = f2fma(kim, sre, f2fma(kre, sim, m[k2].im));
            }
            if (++phx == f) {
                phx = 0;
                ++phy;
            }
        }
        // inverse DFT over k2 and twiddle, then both epochs' values join at column kx and its mirror
        const bool selfcol = kx == 0 || 2 * kx == L;
        float2 *z = pr_dyn + g * ZN + R2Y * k1 * P + ckcol<L>(kx);
        float2 *zm = pr_dyn + g * ZN + R2Y * (k1 == 0 ? 0 : R1Y - k1) * P + ckcol<L>(kx == 0 ? 0 : L - kx);
        zdft<R2Y, true>(m);
        int j = 0;
#pragma unroll
        for (int n2 = 0; n2 < R2Y; ++n2, j += k1) {
            const C2 v = n2 == 0 ? m[0] : zmulwc(m[n2], W[j]);
            z[n2 * P] = make_float2(v.re.x - v.im.y, v.im.x + v.re.y);                 // a + i b
            if (!selfcol) zm[n2 * P] = make_float2(v.re.x + v.im.y, v.re.y - v.im.x);  // conj a + i conj b
        }
    }
    __syncthreads();
}

// Inverse pass A along y of np pairs: rows y = n2 + R2Y n1 < N written.
template <int L>
__device__ __noinline__ void y_inv(int np, int N) {
    using G = Ck<L>;
    constexpr int P = G::P, R1Y = G::R1Y, R2Y = G::R2Y;
    for (int t = threadIdx.x; t < np * R2Y * L; t += blockDim.x) {
        const int c = t % L, r = t / L;
        const int n2 = r % R2Y, g = r / R2Y;
        float2 *z = pr_dyn + g * G::ZN + (c / G::R2X) * G::SX + c % G::R2X + n2 * P;
        float2 v[R1Y];
#pragma unroll
        for (int k1 = 0; k1 < R1Y; ++k1) v[k1] = z[R2Y * k1 * P];
        zdft<R1Y, true>(v);
#pragma unroll
        for (int n1 = 0; n1 < R1Y; ++n1)
            if (n2 + R2Y * n1 < N) z[R2Y * n1 * P] = v[n1];
    }
    __syncthreads();
}

// Forward pass A along y (the twiddle is applied after the epochs are separated).
template <int L>
__device__ __noinline__ void y_fwd(int np, int N) {
    using G = Ck<L>;
    constexpr int P = G::P, R1Y = G::R1Y, R2Y = G::R2Y;
    for (int t = threadIdx.x; t < np * R2Y * L; t += blockDim.x) {
        const int c = t % L, r = t / L;
        const int n2 = r % R2Y, g = r / R2Y;
        float2 *z = pr_dyn + g * G::ZN + (c / G::R2X) * G::SX + c % G::R2X + n2 * P;
        float2 v[R1Y];
#pragma unroll
        for (int n1 = 0; n1 < R1Y; ++n1) v[n1] = n2 + R2Y * n1 < N ? z[R2Y * n1 * P] : make_float2(0.f, 0.f);
        zdft<R1Y, false>(v);
#pragma unroll
        for (int k1 = 0; k1 < R1Y; ++k1) z[R2Y * k1 * P] = v[k1];
    }
    __syncthreads();
}

// Pass B along x of the rows y < N of np pairs (w_off: the roots of unity in pr_dyn).
template <int L, bool INV>
__device__ __noinline__ void x_outer(int np, int N, int w_off) {
    using G = Ck<L>;
    constexpr int R1X = G::R1X, R2X = G::R2X;
    const float2 *W = pr_dyn + w_off;
    const int per = N * R1X;
    const float inv_per = 1.f / (float)per;
    for (int t = threadIdx.x; t < np * per; t += blockDim.x) {
        const int g = np == 1 ? 0 : fdivq(t, inv_per), rem = t - g * per;
        const int row = rem / R1X, k1 = rem - row * R1X;
        float2 *z = pr_dyn + g * G::ZN + row * G::P + k1 * G::SX;
        float2 v[R2X];
#pragma unroll
        for (int q = 0; q < R2X; ++q) v[q] = z[q];
        zdft<R2X, INV>(v);
        int j = 0;
#pragma unroll
        for (int q = 0; q < R2X; ++q, j += k1) z[q] = !INV || q == 0 ? v[q] : zmulwc(v[q], W[j]);
    }
    __syncthreads();
}

// Inverse pass A along x, the residual, forward pass A along x, all on one thread's R1X positions
// x = n2 + R2X n1 of a row; the warps w with w mod np = g take the rows of pair g.  chi^2 and sum e of
// the warp's share of both epochs go to pr_sh.cs.  e is stored halved: the factor of the separation of
// the two epochs' spectra.
template <int L>
__device__ __noinline__ void x_residual(const FieldDev &fd, int i0, int a0, int ne, int w_off) {
    using G = Ck<L>;
    constexpr int R1X = G::R1X, R2X = G::R2X, SX = G::SX;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int N = fd.N, f = fd.f;
    const float2 *W = pr_dyn + w_off;
    const float scale = 1.f / ((float)L * (float)L);
    const unsigned long long pol = l2_policy_first();
    FSum chi[2], se[2];
    chi[0] = chi[1] = se[0] = se[1] = fsum_zero();
    const int np = (ne + 1) / 2;
    const int g = warp % np, sub = warp / np, nsub = (nw - g + np - 1) / np;
    const bool has1 = 2 * g + 1 < ne;
    const float bg0 = (float)(f * f) * pr_sh.ig[a0 + 2 * g], bg1 = has1 ? (float)(f * f) * pr_sh.ig[a0 + 2 * g + 1] : 0.f;
    const float *d0 = fd.d + (long long)(i0 + 2 * g) * N * N, *w0 = fd.w + (long long)(i0 + 2 * g) * N * N;
    const int nn = N * N;
    float2 *zg = pr_dyn + g * G::ZN;
    for (int t = sub * 32 + lane; t < N * R2X; t += nsub * 32) {
        const int row = t / R2X, n2 = t % R2X;
        const float *dr = d0 + row * N + n2, *wr = w0 + row * N + n2;
        float2 dv[R1X], wv[R1X];
#pragma unroll
        for (int n1 = 0; n1 < R1X; ++n1) {
            const bool in = n2 + R2X * n1 < N;
            dv[n1] = wv[n1] = make_float2(0.f, 0.f);
            if (in) {
                dv[n1].x = ldg_hint(dr + R2X * n1, pol);
                wv[n1].x = ldg_hint(wr + R2X * n1, pol);
            }
            if (in && has1) {
                dv[n1].y = ldg_hint(dr + nn + R2X * n1, pol);
                wv[n1].y = ldg_hint(wr + nn + R2X * n1, pol);
            }
        }
        float2 *z = zg + row * G::P + n2;
        float2 v[R1X];
#pragma unroll
        for (int k1 = 0; k1 < R1X; ++k1) v[k1] = z[k1 * SX];
        zdft<R1X, true>(v);
        float2 c = make_float2(0.f, 0.f), sm = make_float2(0.f, 0.f);
#pragma unroll
        for (int n1 = 0; n1 < R1X; ++n1) {
            const float2 r = f2sub(dv[n1], f2fma(v[n1], f2dup(scale), make_float2(bg0, bg1)));
            const float2 wr2 = f2mul(wv[n1], r);  // -e
            c = f2fma(f2mul(wr2, f2dup(0.5f)), r, c);
            sm = f2add(sm, wr2);
            v[n1] = f2mul(wr2, f2dup(-0.5f));
        }
        chi[0] = fsum_add(chi[0], c.x);
        chi[1] = fsum_add(chi[1], c.y);
        se[0] = fsum_add(se[0], -sm.x);
        se[1] = fsum_add(se[1], -sm.y);
        zdft<R1X, false>(v);
        int j = 0;
#pragma unroll
        for (int k1 = 0; k1 < R1X; ++k1, j += n2) z[k1 * SX] = k1 == 0 ? v[0] : zmulw(v[k1], W[j]);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const FSum c = fsum_warp(chi[q]), e = fsum_warp(se[q]);
        if (lane == 0) {
            pr_sh.cs[0][q][warp] = make_float2(c.hi, c.lo);
            pr_sh.cs[1][q][warp] = make_float2(e.hi, e.lo);
        }
    }
    __syncthreads();
}

// The residual spectra (twiddle and forward pass B along y), the adjoint spectra
// acc_phi += sum_e conj(Khat_{e,phi}) ehat_e (pairs and epochs in order) and the sources' Parseval sums
// (a, x, y) per epoch and source into pr_sh.red.  With the column of a unit fixed these factor as
// sum_rows w Re(G conj(gx gy)) = w Re(conj(gx) T1), T1 = sum_rows G conj(gy) (T2 with d gy).  Loads as
// in spec_model.
template <int L, int MS>
__device__ __noinline__ void spec_adjoint(const FieldDev &fd, const float4 *__restrict__ kh, float2 *__restrict__ acc,
                                          int ne, bool first_group, bool last_group, int prof_off, int w_off) {
    using G = Ck<L>;
    constexpr int H = G::H, HP = G::HP, LHP = L * HP, ZN = G::ZN, P = G::P, R1Y = G::R1Y, R2Y = G::R2Y;
    constexpr int UNITS = H * R1Y;
    const int f = fd.f, M = fd.M, nph = f * f, np = (ne + 1) / 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float4 *prof0 = reinterpret_cast<const float4 *>(pr_dyn + prof_off);
    const float2 *W = pr_dyn + w_off;
    const unsigned long long pol_last = l2_policy_last(), pol_first = l2_policy_first();
    for (int g = 0; g < np; ++g) {  // a thread keeps its units, so an accumulator's updates stay in order
        const bool first = first_group && g == 0, last = last_group && g == np - 1;
        float2 sums[MS][3];
#pragma unroll
        for (int k = 0; k < MS; ++k) sums[k][0] = sums[k][1] = sums[k][2] = make_float2(0.f, 0.f);
        for (int t = threadIdx.x; t < UNITS; t += blockDim.x) {
            const int k1 = t / H, kx = t - k1 * H;
            float2 *ac = acc + k1 * HP + kx;
            const float4 *kp = kh + (long long)g * nph * LHP + k1 * HP + kx;
            C2 eh[R2Y];
            {
                const float2 *z = pr_dyn + g * ZN + R2Y * k1 * P + ckcol<L>(kx);
                const float2 *zm = pr_dyn + g * ZN + R2Y * (k1 == 0 ? 0 : R1Y - k1) * P + ckcol<L>(kx == 0 ? 0 : L - kx);
                int j = 0;
#pragma unroll
                for (int n2 = 0; n2 < R2Y; ++n2, j += k1) {
                    const float2 A = z[n2 * P], B = zm[n2 * P];
                    const C2 v{f2add(A, B), make_float2(A.y - B.y, B.x - A.x)};  // A + conj B, (A - conj B) / i
                    eh[n2] = n2 == 0 ? v : zmulw(v, W[j]);
                }
                zdft<R2Y, false>(eh);
            }
            int phy = 0, phx = 0;
            for (int ph = 0; ph < nph; ++ph) {
                float2 av[R2Y];
                float4 kv[R2Y];
#pragma unroll
                for (int k2 = 0; k2 < R2Y; ++k2) {
                    const int off = ph * LHP + k2 * R1Y * HP;
                    av[k2] = first ? make_float2(0.f, 0.f) : ld_hint(ac + off, pol_last);
                    kv[k2] = ldg_hint(kp + off, pol_first);
                }
                const float4 *yt = prof0 + prof_at(g, 0, phy, 2, M, f, H);
                C2 t1[MS], t2[MS];
#pragma unroll
                for (int k = 0; k < MS; ++k) t1[k].re = t1[k].im = t2[k].re = t2[k].im = make_float2(0.f, 0.f);
#pragma unroll
                for (int k2 = 0; k2 < R2Y; ++k2) {
                    const float2 kre = make_float2(kv[k2].x, kv[k2].y), kim = make_float2(kv[k2].z, kv[k2].w);
                    const float2 er = eh[k2].re, ei = eh[k2].im;
                    const float2 gr = f2fma(ei, kim, f2mul(er, kre)), gi = f2nfma(er, kim, f2mul(ei, kre));
                    const float2 run = make_float2((av[k2].x + gr.x) + gr.y, (av[k2].y + gi.x) + gi.y);
                    st_hint(ac + ph * LHP + k2 * R1Y * HP, run, last ? pol_first : pol_last);
                    auto add_t = [&](C2 &tt, float4 y) {  // tt += G conj(y)
                        const float2 yre = make_float2(y.x, y.y), yim = make_float2(y.z, y.w);
                        tt.re = f2fma(gr, yre, tt.re);
                        tt.im = f2fma(gi, yre, tt.im);
                        if (prof_conj<L>(k2)) {
                            tt.re = f2nfma(gi, yim, tt.re);
                            tt.im = f2fma(gr, yim, tt.im);
                        } else {
                            tt.re = f2fma(gi, yim, tt.re);
                            tt.im = f2nfma(gr, yim, tt.im);
                        }
                    };
#pragma unroll
                    for (int k = 0; k < MS; ++k) {
                        if (k < M) {
                            const float4 *y = yt + k * f * 4 * H;
                            add_t(t1[k], prof_val<L>(y, k1, k2));
                            add_t(t2[k], prof_val<L>(y + H, k1, k2));
                        }
                    }
                }
                const float2 wgt = f2dup(kx == 0 || 2 * kx == L ? 1.f : 2.f);  // Parseval weight of the column
#pragma unroll
                for (int k = 0; k < MS; ++k)
                    if (k < M) {
                        const float4 *px = prof0 + prof_at(g, k, phx, 0, M, f, H) + kx;
                        auto dot = [&](const C2 &tt, float4 v) {  // w Re(conj(v) t)
                            return f2mul(wgt, f2fma(tt.im, make_float2(v.z, v.w), f2mul(tt.re, make_float2(v.x, v.y))));
                        };
                        const float4 x = px[0];
                        sums[k][0] = f2add(sums[k][0], dot(t1[k], x));
                        sums[k][1] = f2add(sums[k][1], dot(t1[k], px[H]));
                        sums[k][2] = f2add(sums[k][2], dot(t2[k], x));
                    }
                if (++phx == f) {
                    phx = 0;
                    ++phy;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < MS; ++k) {
            if (k < M) {
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    float2 a = sums[k][q];
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        a.x += __shfl_down_sync(0xffffffffu, a.x, o);
                        a.y += __shfl_down_sync(0xffffffffu, a.y, o);
                    }
                    if (lane == 0) {
                        pr_sh.red[(2 * g * M + k) * 3 + q][warp] = a.x;
                        pr_sh.red[((2 * g + 1) * M + k) * 3 + q][warp] = a.y;
                    }
                }
            }
        }
    }
    __syncthreads();
}

// One item (x = field, y = first epoch, z = end, w = chunk index within the field) in groups of
// fd.fft_G epoch pairs; MS bounds the sources.  The passes are not inlined: each is
// register-allocated on its own.
template <int L, int MS>
__device__ __noinline__ void chunk_item_pair(const FieldDev &fd, const int4 item, const float *__restrict__ params,
                                             const float2 *__restrict__ hhat_all, float2 *__restrict__ acc_all,
                                             double *__restrict__ chi_part, double *__restrict__ se_part,
                                             float *__restrict__ ps_da, float *__restrict__ ps_du) {
    using G = Ck<L>;
    constexpr int LHP = L * G::HP;
    const int GP = fd.fft_G, EG = 2 * GP;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const int f = fd.f, N = fd.N, F = fd.F, M = fd.M, E = fd.E, nph = f * f;
    PrShared &sh = pr_sh;
    const int prof_off = GP * G::ZN, w_off = prof_off + EG * M * f * 4 * G::H;  // tables; W_L^j, j < L
    {
        const float *hpar = params + fd.param_off;
        const float *cpar = hpar + (long long)F * F + (long long)E * M;
        const int n_ep = item.z - item.y;
        for (int j = tid; j < L; j += nt) pr_dyn[w_off + j] = fd.fft_tw[j];
        for (int t = tid; t < n_ep * M; t += nt) sh.ia[t] = hpar[(long long)F * F + (long long)item.y * M + t];
        for (int t = tid; t < 2 * n_ep; t += nt) sh.id[t] = cpar[2 * M + 2 * item.y + t];
        for (int t = tid; t < n_ep; t += nt) sh.ig[t] = cpar[2 * M + 2 * E + item.y + t];
        for (int t = tid; t < 2 * M; t += nt) sh.ic[t] = cpar[t];
    }
    __syncthreads();
    const float2 *hh = hhat_all + fd.fft_hhat_off;
    float2 *acc = acc_all + fd.fft_acc_off + (long long)item.w * nph * LHP;
    for (int i0 = item.y; i0 < item.z; i0 += EG) {
        const int ne = min(EG, item.z - i0), a0 = i0 - item.y;
        const int np = (ne + 1) / 2;
        const float4 *kh = reinterpret_cast<const float4 *>(fd.fft_khat) + (long long)(i0 / 2) * nph * LHP;
        // The next group's data and weights go to L2 while this one computes (sizes are multiples of
        // 16 bytes when N is even).  The kernel spectra are not prefetched: with every SM streaming
        // its own group's spectra, an early copy in L2 is evicted before its use (measured slower).
        if (tid == 0 && i0 + EG < item.z && (N & 1) == 0) {
            const int nn = min(EG, item.z - i0 - EG);
            prefetch_l2(fd.d + (long long)(i0 + EG) * N * N, (long long)nn * N * N * 4);
            prefetch_l2(fd.w + (long long)(i0 + EG) * N * N, (long long)nn * N * N * 4);
        }
        if (M > 0) window_profiles<L>(fd, sh, a0, ne, np, pr_dyn, reinterpret_cast<float4 *>(pr_dyn + prof_off), pr_dyn + w_off);
        __syncthreads();
        spec_model<L, MS>(fd, hh, kh, a0, ne, prof_off, w_off);
        y_inv<L>(np, N);
        x_outer<L, true>(np, N, w_off);
        x_residual<L>(fd, i0, a0, ne, w_off);
        x_outer<L, false>(np, N, w_off);
        y_fwd<L>(np, N);
        spec_adjoint<L, MS>(fd, kh, acc, ne, i0 == item.y, i0 + EG >= item.z, prof_off, w_off);
        // warp v sums value v's per-warp partials in a fixed shuffle tree
        const int nv = 2 + 3 * M;
        for (int v = warp; v < ne * nv; v += nw) {
            const int e = v / nv, q = v - e * nv;
            float2 part = make_float2(0.f, 0.f);
            if (lane < nw) {
                if (q >= 2) part.x = sh.red[e * 3 * M + q - 2][lane];
                else if (lane % np == e / 2) part = sh.cs[q][e & 1][lane];
            }
            const FSum tot = fsum_warp(FSum{part.x, part.y});
            if (lane == 0) {
                const double sum = fsum_value(tot);
                const int i = i0 + e;
                if (q == 0) {
                    chi_part[fd.tile_slot + i] = sum;
                } else if (q == 1) {
                    se_part[fd.tile_slot + i] = sum;
                } else {
                    constexpr double kInvL2 = 1.0 / ((double)L * (double)L);
                    const int k = (q - 2) / 3, which = (q - 2) - 3 * k;
                    const long long ps = fd.ps_slot + (long long)i * M + k;
                    const float sc = (float)(sum * kInvL2);
                    if (which == 0) ps_da[ps] = sc;
                    else ps_du[2 * ps + which - 1] = sh.ia[(a0 + e) * M + k] * sc;
                }
            }
        }
        __syncthreads();
    }
}

template <int L>
__device__ __forceinline__ void chunk_item_dispatch(const FieldDev &fd, const int4 item, const float *params,
                                                    const float2 *hhat, float2 *acc, double *chi_part,
                                                    double *se_part, float *ps_da, float *ps_du) {
    if (fd.M > 1)
        chunk_item_pair<L, kFftMaxSources>(fd, item, params, hhat, acc, chi_part, se_part, ps_da, ps_du);
    else
        chunk_item_pair<L, 1>(fd, item, params, hhat, acc, chi_part, se_part, ps_da, ps_du);
}

__global__ void __launch_bounds__(kChunkThreads, 1)
fft_chunk_pair_kernel(const FieldDev *__restrict__ fields, const int4 *__restrict__ items, int n_items,
                      int *__restrict__ counter, const float *__restrict__ params, const float2 *__restrict__ hhat_all,
                      float2 *__restrict__ acc_all, double *__restrict__ chi_part, double *__restrict__ se_part,
                      float *__restrict__ ps_da, float *__restrict__ ps_du) {
    for (;;) {
        if (threadIdx.x == 0) pr_sh.item = atomicAdd(counter, 1);
        __syncthreads();
        const int it = pr_sh.item;
        if (it >= n_items) break;
        const int4 item = items[it];
        const FieldDev &fd = fields[item.x];
        switch (fd.fft_L) {
#define SR_PR_CASE(LL)                                                                                      \
    case LL:                                                                                                \
        chunk_item_dispatch<LL>(fd, item, params, hhat_all, acc_all, chi_part, se_part, ps_da, ps_du);      \
        break;
            SR_PR_SIZES(SR_PR_CASE)
#undef SR_PR_CASE
            default:
                break;  // not reached: the host only builds items for sizes in the list
        }
        __syncthreads();
    }
}

template <int L>
constexpr int pair_zn() {
    return Pr<L>::ZN;
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
bool fft_pair_size(int L) {
    switch (L) {
#define SR_PR_OK(LL) case LL:
        SR_PR_SIZES(SR_PR_OK)
#undef SR_PR_OK
        return true;
        default:
            return false;
    }
}

int fft_pair_next(int need) {
    static const int sizes[] = {
#define SR_PR_LIST(LL) LL,
        SR_PR_SIZES(SR_PR_LIST)
#undef SR_PR_LIST
    };
    for (int L : sizes)
        if (L >= need) return L;
    return 0;
}

int fft_pair_zn(int L) {
    switch (L) {
#define SR_PR_ZN(LL) \
    case LL:         \
        return pair_zn<LL>();
        SR_PR_SIZES(SR_PR_ZN)
#undef SR_PR_ZN
        default:
            return 0;
    }
}

int fft_pair_smem_bytes(int L, int M, int f, int GP) {
    switch (L) {
#define SR_PR_SM(LL) \
    case LL:         \
        return ck_smem<LL>(GP, M, f);
        SR_PR_SIZES(SR_PR_SM)
#undef SR_PR_SM
        default:
            return 0;
    }
}

// The per-field and per-PSF kernels: one pair array and the twiddles.
int fft_pair_field_smem(int L) { return (fft_pair_zn(L) + L) * (int)sizeof(float2); }

// Epoch pairs per group of the chunk kernel at size L with at most one source, else 1.
int fft_pair_gpmax(int L, int M) {
    if (M > 1) return 1;
    switch (L) {
#define SR_PR_GM(LL) \
    case LL:         \
        return pr_gpmax<LL>();
        SR_PR_SIZES(SR_PR_GM)
#undef SR_PR_GM
        default:
            return 1;
    }
}

// Epoch pairs side by side: the widest group the kernel is compiled for at this size (more than one pair
// only with at most one source) if its buffers fit, else one pair.
int fft_pair_group(int L, int M, int f, int gp_cap, int smem_limit) {
    const int G = gp_cap != 1 ? fft_pair_gpmax(L, M) : 1;
    return G > 1 && fft_pair_smem_bytes(L, M, f, G) > smem_limit ? 1 : G;
}

// Default epochs per work item of the transform form (even, 2 .. kFftChunk): the shortest time to
// finish the items on one block per SM, longest first, plus the traffic of their accumulators.
// An item costs its epoch pairs' transforms (measured: 8 to 11 cycles per point of the L x L pair at
// f = 2, by the phases above that, and 0.45 more per further source; 0.6 of it once per group of pairs,
// whose passes it shares) and a fixed part; an accumulator is written, read back and added at about
// 400 bytes a clock over the GPU.  Against "as many epochs as keep two items per SM" (us per evaluation):
// 1000 epochs of 32 x 32 157 -> 102 (8 epochs instead of 2: 125 items finish together, 500 leave a fourth of
// a round and 4 times the accumulators), 500 of 48 x 48 123 -> 94, 24 fields of 10-60 epochs 269 -> 193; 300 of 64 x 64 keeps 2, 300 of 88 x 88 at f =
// 3, whose buffers leave room for one pair, take 2 (193; 222 with the 4 of two pairs).  Groups capped to one pair by
// the caller keep the epochs of the widest (1000 of 24 x 24: 104 with 8, 126 with the 4 of that pricing).  Fields
// that fill the GPU several times at the longest items take those.
int fft_chunk_epochs(const FftShape *shapes, int n, int n_sms, int smem_limit) {
    struct Shape {
        double pair, acc;  // cycles of a pair; accumulator bytes
        int epochs, group;
    };
    std::vector<Shape> sh;
    long long longest = 0;
    for (int i = 0; i < n; ++i) {
        const FftShape &p = shapes[i];
        const double L = p.L, nph = (double)p.f * p.f;
        sh.push_back({9.0 * L * L * (0.25 + 0.1875 * nph) * (1.0 + 0.45 * std::max(0, p.M - 1)),
                      nph * L * (L / 2 + 2) * 8.0, p.E, fft_pair_group(p.L, p.M, p.f, 0, smem_limit)});
        longest += (p.E + kFftChunk - 1) / kFftChunk;
    }
    if (longest >= 4LL * n_sms) return kFftChunk;
    std::stable_sort(sh.begin(), sh.end(), [](const Shape &a, const Shape &b) { return a.pair > b.pair; });
    int best = 2;
    double best_t = 0.0;
    for (int c = 2; c <= kFftChunk; c += 2) {
        std::vector<double> items;
        double bytes = 0.0;
        for (const Shape &s : sh)
            for (int e = 0; e < s.epochs; e += c) {
                const int pairs = (std::min(c, s.epochs - e) + 1) / 2, groups = (pairs + s.group - 1) / s.group;
                items.push_back((0.6 * groups + 0.4 * pairs) * s.pair + 4000.0);
                bytes += 2.0 * s.acc;
            }
        std::sort(items.begin(), items.end(), [](double a, double b) { return a > b; });
        std::priority_queue<double, std::vector<double>, std::greater<double>> free_at;
        double end = 0.0;
        for (double t : items) {
            double at = 0.0;
            if ((int)free_at.size() >= n_sms) {
                at = free_at.top();
                free_at.pop();
            }
            free_at.push(at + t);
            end = std::max(end, at + t);
        }
        const double total = end + bytes / 400.0;
        if (c == 2 || total < std::min(0.95 * best_t, best_t - 20000.0)) {  // 10 us at least
            best = c;
            best_t = total;
        }
    }
    return best;
}

// Whether the chunk kernel takes M sources at size L (one pair per group, two phases).
bool fft_pair_variant(int L, int M) {
    return fft_pair_size(L) && M <= kFftMaxSources &&
           (M <= 1 || fft_pair_smem_bytes(L, kFftMaxSources, 2, 1) <= kChunkSmem);
}

template <typename K>
static sr_status open_smem(K kernel, int optin, int *limit) {
    cudaFuncAttributes a;
    SR_CUDA(cudaFuncGetAttributes(&a, kernel));
    const int dyn = optin - (int)a.sharedSizeBytes;
    SR_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn));
    *limit = std::min(*limit, dyn);
    return SR_OK;
}

// Fills the DFT twiddle tables and opens the largest dynamic shared memory each kernel can take;
// *chunk_limit and *field_limit are what the chunk kernel and the per-field kernels may use.
sr_status configure_fft_pair(int optin, int *chunk_limit, int *field_limit) {
    SR_CUDA(pr_fill_dtw());
    *chunk_limit = optin;
    sr_status s;
    if ((s = open_smem(fft_chunk_pair_kernel, optin, chunk_limit)) != SR_OK) return s;
    return configure_fft_pair_field(optin, field_limit);
}


sr_status occupancy_fft_pair(int smem, int *blocks) {
    SR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, fft_chunk_pair_kernel, kChunkThreads, smem));
    return SR_OK;
}

void launch_fft_chunks_pair(const FieldDev *fields, const int4 *items, int n_items, int *counter, const float *params,
                            const float2 *hhat, float2 *acc, double *chi_part, double *se_part, float *ps_da,
                            float *ps_du, int grid, int smem, cudaStream_t st) {
    fft_chunk_pair_kernel<<<grid, kChunkThreads, smem, st>>>(fields, items, n_items, counter, params, hhat, acc,
                                                           chi_part, se_part, ps_da, ps_du);
}

}  // namespace sr
