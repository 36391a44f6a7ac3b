// Noise propagation to the starlet coefficients (sec. 2.3, App. B): the prior weights W by
// Monte Carlo.
//
// Realisation r draws a standard normal field z_r on the fine grid, forms
// (C^)^-1 dd = z_r / sigma_eff^ (the co-added noise map, sigma_eff^-2 = sum_i sigma_i^-2,
// replicated over the f x f fine pixels of each data pixel), applies S_1^T (correlation with
// epoch 1's narrow PSF, the transpose of the zero-padded "same" convolution) and the starlet
// analysis.  W_j is the standard deviation of the detail plane w_{j+1}: per coefficient over
// the realisations (the map), and pooled over the plane's coefficients and the realisations
// (the one number per scale that the prior takes).
//
// Random numbers: normal number n of stream `seed` comes from Philox4x64-10 (Salmon et al.
// 2011) block n/4 with counter (n/4, 0, 0, 0) and key (seed, 0); the block's words (0,1) and
// (2,3) give two Box-Muller pairs from 24-bit uniforms u = ((w >> 40) + 1) 2^-24, cos then sin.
// Realisation r uses the numbers r F^2 .. r F^2 + F^2 - 1 in row-major pixel order.
//
// Work per batch of B realisations (all resident in L2):
//   noise_draw_kernel      x[b]  = z / sigma_eff^                     (one Philox block a thread)
//   noise_corr_kernel      y[b]  = S_1^T x[b]                          (FP32, 2 F^2 K^2 flop each), or
//   noise_fft_kernel       the same by transforms (noise_fft.cu), where that is cheaper and as accurate
//                          (noise_level, in the first batch's draw, tells; if not, the call starts over
//                          with the direct form)
//   noise_row_kernel       t[b]  = row pass of level j on c_j[b]
//   noise_col_stats_kernel c_{j+1}[b] = column pass; w = c_j - c_{j+1}; sum and sum of squares of
//                          w over the batch, in a fixed order, into per-segment FP64 accumulators
// and at the end noise_map_kernel / noise_scale_kernel reduce the segments in a fixed order.
// The direct correlation is bound by FP32 FMA issue (5000 realisations at F = 128, K = 64: 11.7 ms);
// with the transforms (0.78 ms) the column passes are the largest part.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "ffsum.cuh"
#include "noise.cuh"

namespace sr {
namespace {

// ---- counter-based normals ---------------------------------------------------------------

constexpr uint64_t kPhM0 = 0xD2E7470EE14C6C93ULL, kPhM1 = 0xCA5A826395121157ULL;
constexpr uint64_t kPhW0 = 0x9E3779B97F4A7C15ULL, kPhW1 = 0xBB67AE8584CAA73BULL;

__device__ __forceinline__ void philox4x64_10(uint64_t &c0, uint64_t &c1, uint64_t &c2, uint64_t &c3, uint64_t k0,
                                              uint64_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t hi0 = __umul64hi(kPhM0, c0), lo0 = kPhM0 * c0;
        const uint64_t hi1 = __umul64hi(kPhM1, c2), lo1 = kPhM1 * c2;
        const uint64_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
        k0 += kPhW0;
        k1 += kPhW1;
    }
}

__device__ __forceinline__ float uniform24(uint64_t w) { return (float)((w >> 40) + 1) * 0x1p-24f; }

// x[b][u] = z(seed, (r0 + b) F^2 + u) * isig[u] for the n = B F^2 numbers of the batch.  The batch
// starts at pixel 0 of its first realisation, so the pixel of number n0 + i is i mod F^2, in 32 bits
// (Int) unless one realisation alone is larger than that: a 64-bit remainder per number cost as much
// as the generator (5000 realisations at F = 128: 0.53 ms before, 0.43 ms with this).
// Block b of nb.
template <typename Int>
__device__ __forceinline__ void noise_draw(const float *__restrict__ isig, int F, uint64_t seed, long long r0, int B,
                                           float *__restrict__ x, int b, int nb) {
    const Int FF = (Int)F * F;
    const long long n0 = r0 * FF;
    const Int total = B * FF;
    const int lead = (int)(n0 & 3);  // the first block's numbers before the batch
    const long long blk0 = n0 >> 2;
    const Int nblk = (lead + total + 3) >> 2;
    for (Int k = b * (int)blockDim.x + (int)threadIdx.x; k < nblk; k += nb * (int)blockDim.x) {
        uint64_t c0 = (uint64_t)(blk0 + k), c1 = 0, c2 = 0, c3 = 0;
        philox4x64_10(c0, c1, c2, c3, seed, 0);
        float z[4];
        {
            const float r = sqrtf(-2.f * logf(uniform24(c0)));
            float s, c;
            sincospif(2.f * uniform24(c1), &s, &c);
            z[0] = r * c;
            z[1] = r * s;
        }
        {
            const float r = sqrtf(-2.f * logf(uniform24(c2)));
            float s, c;
            sincospif(2.f * uniform24(c3), &s, &c);
            z[2] = r * c;
            z[3] = r * s;
        }
        const Int i0 = 4 * k - lead;
        Int u = (i0 < 0 ? 0 : i0) % FF;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const Int i = i0 + e;
            if (i < 0 || i >= total) continue;
            x[i] = z[e] * isig[u];
            if (++u == FF) u = 0;
        }
    }
}

// ---- S_1^T: zero-padded correlation, register-blocked ---------------------------------------
//
// y[v] = sum_{qy,qx} s[qy][qx] x[vy + qy - o][vx + qx - o]   (o = K/2; x = 0 outside the grid)
//
// A block of kCorrWarps warps computes a TY x TX tile of one realisation.  Lane l of warp w
// owns output rows w*2*RY + (l/16)*RY + i (i < RY) and the two column groups 4(l%16) + j and
// 64 + 4(l%16) + j (j < 4).  The kernel rows are taken KC at a time (KC >= RY): the x rows the
// chunk needs ((TY + KC - 1) x (TX + KP), zero-filled outside the grid) and the chunk's kernel
// rows (zero beyond K) are staged in shared memory.  For x row r of the thread's window, output
// row i uses kernel row r - i, so rows r < RY - 1 and r >= KC feed only part of the RY outputs:
// corr_row takes the range of i as template arguments and no FMA is spent on a missing row.
// Per group of four kernel columns, two float4 of x (a quarter-warp reads 128 consecutive
// bytes: no bank conflict) and one broadcast float4 of s per output row feed 32 FMAs per row;
// the FMAs are ordered by kernel column so that consecutive ones share their s operand.

constexpr int kCorrRY = 4;
constexpr int kCorrWarps = 4;
constexpr int kCorrTY = 2 * kCorrRY * kCorrWarps;  // 32 output rows per block
constexpr int kCorrTX = 128;                       // 16 column groups x 2 x 4 columns
constexpr int kCorrThreads = 32 * kCorrWarps;
constexpr int kCorrMinBlocks = 3;                  // blocks per SM the chunk size aims for

size_t corr_smem_bytes(int KP, int KC) {
    return sizeof(float) * ((size_t)(kCorrTY + KC - 1) * (kCorrTX + KP) + (size_t)KC * KP);
}

// x row r of the window against kernel rows r - i for i in [ILO, IHI)
template <int ILO, int IHI>
__device__ __forceinline__ void corr_row(float (&acc)[kCorrRY][2][4], const float4 *__restrict__ xp,
                                         const float *__restrict__ ss, int r, int KP) {
    const int G = KP / 4;
    float4 A0 = xp[0], A1 = xp[16];
#pragma unroll 4
    for (int g = 0; g < G; ++g) {
        const float4 B0 = xp[g + 1], B1 = xp[g + 17];
        const float xa[2][8] = {{A0.x, A0.y, A0.z, A0.w, B0.x, B0.y, B0.z, B0.w},
                                {A1.x, A1.y, A1.z, A1.w, B1.x, B1.y, B1.z, B1.w}};
#pragma unroll
        for (int i = ILO; i < IHI; ++i) {
            const float4 sv = reinterpret_cast<const float4 *>(ss + (size_t)(r - i) * KP)[g];
            const float se[4] = {sv.x, sv.y, sv.z, sv.w};
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][h][j] = fmaf(se[e], xa[h][j + e], acc[i][h][j]);
        }
        A0 = B0;
        A1 = B1;
    }
}

__global__ void __launch_bounds__(kCorrThreads, kCorrMinBlocks)
    noise_corr_kernel(const float *__restrict__ x, const float *__restrict__ s, int F, int K, int KP, int KC,
                      float *__restrict__ y) {
    static_assert(kCorrRY == 4, "the head and tail rows below are written out for RY = 4");
    extern __shared__ float4 corr_sm4[];
    const int XR = kCorrTY + KC - 1, XW = kCorrTX + KP;
    float *xs = reinterpret_cast<float *>(corr_sm4);
    float *ss = xs + (size_t)XR * XW;
    const int b = blockIdx.z, ty0 = blockIdx.y * kCorrTY, tx0 = blockIdx.x * kCorrTX;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, o = K / 2;
    const int row0 = warp * 2 * kCorrRY + (lane >> 4) * kCorrRY, col0 = 4 * (lane & 15);
    const float *xb = x + (size_t)b * F * F;

    float acc[kCorrRY][2][4];
#pragma unroll
    for (int i = 0; i < kCorrRY; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][0][j] = acc[i][1][j] = 0.f;

    for (int q0 = 0; q0 < K; q0 += KC) {
        __syncthreads();
        for (int idx = threadIdx.x; idx < XR * XW; idx += kCorrThreads) {
            const int t = idx / XW, c = idx - t * XW;
            const int gy = ty0 - o + q0 + t, gx = tx0 - o + c;
            xs[idx] = (gy >= 0 && gy < F && gx >= 0 && gx < F) ? xb[(size_t)gy * F + gx] : 0.f;
        }
        for (int idx = threadIdx.x; idx < KC * KP; idx += kCorrThreads) {
            const int qy = idx / KP, qx = idx - qy * KP, q = q0 + qy;
            ss[idx] = (q < K && qx < K) ? s[(size_t)q * K + qx] : 0.f;
        }
        __syncthreads();
        const float *xrow = xs + (size_t)row0 * XW + col0;
        auto xp = [&](int r) { return reinterpret_cast<const float4 *>(xrow + (size_t)r * XW); };
        corr_row<0, 1>(acc, xp(0), ss, 0, KP);
        corr_row<0, 2>(acc, xp(1), ss, 1, KP);
        corr_row<0, 3>(acc, xp(2), ss, 2, KP);
        for (int r = kCorrRY - 1; r < KC; ++r) corr_row<0, kCorrRY>(acc, xp(r), ss, r, KP);
        corr_row<1, 4>(acc, xp(KC), ss, KC, KP);
        corr_row<2, 4>(acc, xp(KC + 1), ss, KC + 1, KP);
        corr_row<3, 4>(acc, xp(KC + 2), ss, KC + 2, KP);
    }
    float *yb = y + (size_t)b * F * F;
#pragma unroll
    for (int i = 0; i < kCorrRY; ++i) {
        const int vy = ty0 + row0 + i;
        if (vy >= F) break;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int vx = tx0 + 64 * h + col0 + j;
                if (vx < F) yb[(size_t)vy * F + vx] = acc[i][h][j];
            }
    }
}

// ---- batched starlet analysis with per-coefficient moments ---------------------------------

constexpr float kH0 = 0.0625f, kH1 = 0.25f, kH2 = 0.375f;  // B3 spline (1,4,6,4,1)/16

__device__ __forceinline__ int reflect(int t, int F) { return t < 0 ? -t : (t > F - 1 ? 2 * (F - 1) - t : t); }

// t[b][y][x] = sum_m h[m] c[b][y][reflect(x + m step)]
__global__ void __launch_bounds__(256) noise_row_kernel(const float *__restrict__ c, float *__restrict__ t, int F,
                                                        int step, long long total, const int *__restrict__ skip) {
    if (skip && *skip) return;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < total;
         idx += (long long)gridDim.x * blockDim.x) {
        const int xx = (int)(idx % F);
        const float *row = c + (idx - xx);
        t[idx] = kH0 * (row[reflect(xx - 2 * step, F)] + row[reflect(xx + 2 * step, F)]) +
                 kH1 * (row[reflect(xx - step, F)] + row[reflect(xx + step, F)]) + kH2 * row[xx];
    }
}

// Column pass of level j for the realisations of segment blockIdx.y, pixel u per thread:
// c_{j+1} = column filter of t, w = c_j - c_{j+1} (c updated in place: only this thread reads or
// writes c[b][u]); the segment's sums of w and w^2, taken over b in increasing order (groups of
// four in FP32, the groups as compensated pairs), are added to acc1/acc2[seg][j][u].
__global__ void __launch_bounds__(256) noise_col_stats_kernel(float *__restrict__ c, const float *__restrict__ t,
                                                              int F, int step, int B, int S, int J1, int j,
                                                              double *__restrict__ acc1, double *__restrict__ acc2) {
    const long long FF = (long long)F * F;
    const long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (u >= FF) return;
    const int seg = blockIdx.y;
    const int b0 = (int)((long long)B * seg / S), b1 = (int)((long long)B * (seg + 1) / S);
    const int yy = (int)(u / F), xx = (int)(u - (long long)yy * F);
    const long long o_m2 = (long long)reflect(yy - 2 * step, F) * F + xx, o_p2 = (long long)reflect(yy + 2 * step, F) * F + xx;
    const long long o_m1 = (long long)reflect(yy - step, F) * F + xx, o_p1 = (long long)reflect(yy + step, F) * F + xx;
    FSum s1 = fsum_zero(), s2 = fsum_zero();
    int b = b0;
    for (; b + 4 <= b1; b += 4) {  // four realisations' loads issued before their arithmetic
        float tv[4][5], cv[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float *tb = t + (b + k) * FF;
            tv[k][0] = tb[o_m2];
            tv[k][1] = tb[o_m1];
            tv[k][2] = tb[u];
            tv[k][3] = tb[o_p1];
            tv[k][4] = tb[o_p2];
            cv[k] = c[(b + k) * FF + u];
        }
        // the four realisations summed in FP32 (in order), then added to the segment's sums as
        // compensated FP32 pairs (48 significand bits; FP64 additions run at 2 a clock per SM and
        // took a fifth of the column passes: 2.4 -> 1.95 ms per 5000 realisations at F = 128, J = 4)
        float q1 = 0.f, q2 = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float cn = kH0 * (tv[k][0] + tv[k][4]) + kH1 * (tv[k][1] + tv[k][3]) + kH2 * tv[k][2];
            const float w = cv[k] - cn;
            c[(b + k) * FF + u] = cn;
            q1 += w;
            q2 = fmaf(w, w, q2);
        }
        s1 = fsum_add(s1, q1);
        s2 = fsum_add(s2, q2);
    }
    for (; b < b1; ++b) {
        const float *tb = t + b * FF;
        const float cn = kH0 * (tb[o_m2] + tb[o_p2]) + kH1 * (tb[o_m1] + tb[o_p1]) + kH2 * tb[u];
        float *cb = c + b * FF + u;
        const float w = *cb - cn;
        *cb = cn;
        s1 = fsum_add(s1, w);
        const float w2 = w * w;
        s2 = fsum_add(s2, FSum{w2, fmaf(w, w, -w2)});
    }
    const long long k = ((long long)seg * J1 + j) * FF + u;
    acc1[k] += fsum_value(s1);
    acc2[k] += fsum_value(s2);
}

// W_map[j][u] = sample std (n - 1) of w_{j+1}[u] over the n realisations (segments summed in order).
__global__ void __launch_bounds__(256) noise_map_kernel(const double *__restrict__ acc1,
                                                        const double *__restrict__ acc2, long long per_seg, int S,
                                                        int n, float *__restrict__ W_map) {
    const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (k >= per_seg) return;
    double t1 = 0.0, t2 = 0.0;
    for (int s = 0; s < S; ++s) {
        t1 += acc1[s * per_seg + k];
        t2 += acc2[s * per_seg + k];
    }
    const double mean = t1 / n, var = (t2 - n * mean * mean) / (n - 1);
    W_map[k] = (float)sqrt(var > 0.0 ? var : 0.0);
}

// W_scale[j] = sample std (n F^2 - 1) of every coefficient of plane j, in two fixed-shape steps:
// block (b, j) sums its share of the plane's pixels over the segments, and the last block of the
// plane to finish (counted in done[j], zero before the launch) adds the blocks' partials.  (One block per plane took 0.30 ms at F = 128: its loads are a single chain
// of 64 x 16 per thread.)
constexpr int kScaleThreads = 256, kScaleBlocks = 64;
__global__ void __launch_bounds__(kScaleThreads) noise_scale_kernel(const double *__restrict__ acc1,
                                                                    const double *__restrict__ acc2, long long FF,
                                                                    int J1, int S, int n, double2 *part, int *done,
                                                                    float *__restrict__ W) {
    __shared__ double r1[kScaleThreads], r2[kScaleThreads];
    __shared__ bool s_last;
    const int j = blockIdx.y;
    const long long per_seg = FF * J1;
    double t1 = 0.0, t2 = 0.0;
    for (long long u = blockIdx.x * (long long)kScaleThreads + threadIdx.x; u < FF; u += kScaleBlocks * kScaleThreads)
#pragma unroll 4
        for (int s = 0; s < S; ++s) {
            t1 += acc1[s * per_seg + j * FF + u];
            t2 += acc2[s * per_seg + j * FF + u];
        }
    r1[threadIdx.x] = t1;
    r2[threadIdx.x] = t2;
    __syncthreads();
    for (int h = kScaleThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            r1[threadIdx.x] += r1[threadIdx.x + h];
            r2[threadIdx.x] += r2[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[j * kScaleBlocks + blockIdx.x] = make_double2(r1[0], r2[0]);
        __threadfence();
        s_last = atomicAdd(&done[j], 1) == kScaleBlocks - 1;
    }
    __syncthreads();
    if (!s_last || threadIdx.x >= 32) return;
    __threadfence();
    t1 = t2 = 0.0;
    for (int b = threadIdx.x; b < kScaleBlocks; b += 32) {
        const double2 v = __ldcg(&part[j * kScaleBlocks + b]);
        t1 += v.x;
        t2 += v.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        t1 += __shfl_down_sync(0xffffffffu, t1, o);
        t2 += __shfl_down_sync(0xffffffffu, t2, o);
    }
    if (threadIdx.x == 0) {
        const double m = (double)n * (double)FF, mean = t1 / m, var = (t2 - m * mean * mean) / (m - 1.0);
        W[j] = (float)sqrt(var > 0.0 ? var : 0.0);
    }
}

// The set-up of a call, one launch:
// blocks [0, n_isig): 1/sigma_eff on the fine grid; flags (bit 0) a NaN or non-positive sigma and
//   (bit 1) a non-finite PSF value.  A block takes 32 data pixels (lanes) and deals the epochs over
//   its 8 warps (epoch i to warp i mod 8, the warps' sums added in order), so that the epochs' loads
//   are in flight together; one thread per fine pixel walking every epoch took 0.25 ms at E = 300,
//   N = 64.
// blocks n_isig + kx, kx < spec.L: column kx of the transform form's kernel spectrum (noise_spectrum).
// block n_isig + spec.L, with spec.L > 0: the PSF's norm and peak (noise_peak).
constexpr int kIsigWarps = 8;

__device__ void noise_isig(const float *__restrict__ sigma, const float *__restrict__ s1, int N, int f, int E, int K,
                           int n_blocks, float *__restrict__ isig, int *__restrict__ flag,
                           double (*part)[32]) {
    const int F = f * N, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long NN = (long long)N * N, KK = (long long)K * K;
    for (long long u = blockIdx.x * (long long)blockDim.x + threadIdx.x; u < KK; u += (long long)n_blocks * blockDim.x)
        if (!isfinite(s1[u])) atomicOr(flag, 2);
    for (long long p0 = blockIdx.x * 32LL; p0 < NN; p0 += n_blocks * 32LL) {
        const long long p = p0 + lane;
        double iv = 0.0;
        bool bad = false;
        if (p < NN) {
#pragma unroll 4
            for (int i = warp; i < E; i += kIsigWarps) {
                const float sg = __ldg(sigma + i * NN + p);
                if (isnan(sg) || sg <= 0.f) bad = true;
                else if (isfinite(sg)) iv += 1.0 / ((double)sg * (double)sg);
            }
        }
        if (bad) atomicOr(flag, 1);
        part[warp][lane] = iv;
        __syncthreads();
        if (warp == 0 && p < NN) {
            double t = 0.0;
            for (int w = 0; w < kIsigWarps; ++w) t += part[w][lane];
            const float v = (float)sqrt(t);
            const int py = (int)(p / N), px = (int)(p - (long long)py * N);
            for (int ay = 0; ay < f; ++ay)
                for (int ax = 0; ax < f; ++ax) isig[(long long)(f * py + ay) * F + f * px + ax] = v;
        }
        __syncthreads();
    }
}

// Column kx of conj(Shat) / L^2 = L^-2 sum_{q,t} s[q][t] exp(2 pi i (ky (q - sh) + kx (t - sh)) / L),
// summed over t, then over q, in FP64 and rounded once, at [position of ky][position of kx] of the
// transforms' digit-transposed order (position R2 (k mod R1) + k / R1), divided by the gains of both
// axes; kx = 0 also writes the twiddles exp(-2 pi i j / L).
constexpr int kSpecMax = 256;
__device__ void noise_spectrum(const float *__restrict__ s, int K, int kx, const NoiseSpec &sp, double2 *w, double2 *R) {
    const int L = sp.L, R2 = L / sp.R1;
    for (int j = threadIdx.x; j < L; j += blockDim.x) {
        double si, co;
        sincospi(2.0 * (double)j / (double)L, &si, &co);
        w[j] = make_double2(co, si);
        if (kx == 0) sp.tw[j] = make_float2((float)co, (float)-si);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < K; q += blockDim.x) {
        double a = 0.0, b = 0.0;
        int j = (int)((long long)kx * (L - sp.sh) % L);
        for (int t = 0; t < K; ++t) {
            const double v = (double)__ldg(s + (long long)q * K + t);
            a += v * w[j].x;
            b += v * w[j].y;
            j += kx;
            if (j >= L) j -= L;
        }
        R[q] = make_double2(a, b);
    }
    __syncthreads();
    const double scale = 1.0 / ((double)L * (double)L * sp.gain[kx]);  // and by gain[ky] below
    const int pc = R2 * (kx % sp.R1) + kx / sp.R1;
    for (int ky = threadIdx.x; ky < L; ky += blockDim.x) {
        double a = 0.0, b = 0.0;
        int j = (int)((long long)ky * (L - sp.sh) % L);
        for (int q = 0; q < K; ++q) {
            a += R[q].x * w[j].x - R[q].y * w[j].y;
            b += R[q].x * w[j].y + R[q].y * w[j].x;
            j += ky;
            if (j >= L) j -= L;
        }
        const double sc = scale / sp.gain[ky];
        sp.S[(long long)(R2 * (ky % sp.R1) + ky / sp.R1) * L + pc] = make_float2((float)(a * sc), (float)(b * sc));
    }
}

// Norm^2 and position of the largest |s| (the first of equals), by one block.
struct NoisePeak {
    double norm2;
    int qy, qx;
};
__device__ void noise_peak(const float *__restrict__ s, int K, NoisePeak *peak, double2 *red) {
    double n2 = 0.0, top = -1.0;
    int at = 0;
    for (int q = threadIdx.x; q < K * K; q += blockDim.x) {
        const double v = (double)__ldg(s + q);
        n2 += v * v;
        if (fabs(v) > top) {
            top = fabs(v);
            at = q;
        }
    }
    __shared__ int s_at[kSpecMax];
    red[threadIdx.x] = make_double2(n2, top);
    s_at[threadIdx.x] = at;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            const double2 a = red[threadIdx.x], b = red[threadIdx.x + w];
            const int ia = s_at[threadIdx.x], ib = s_at[threadIdx.x + w];
            const bool other = b.y > a.y || (b.y == a.y && ib < ia);
            red[threadIdx.x] = make_double2(a.x + b.x, other ? b.y : a.y);
            s_at[threadIdx.x] = other ? ib : ia;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) *peak = NoisePeak{red[0].x, s_at[0] / K, s_at[0] % K};
}

__global__ void __launch_bounds__(32 * kIsigWarps)
noise_setup_kernel(const float *__restrict__ sigma, const float *__restrict__ s1, int N, int f, int E, int K,
                   int n_isig, float *__restrict__ isig, int *__restrict__ flag, NoiseSpec spec, NoisePeak *peak) {
    __shared__ double2 w[kSpecMax], R[kSpecMax];
    if ((int)blockIdx.x < n_isig)
        noise_isig(sigma, s1, N, f, E, K, n_isig, isig, flag, reinterpret_cast<double (*)[32]>(w));
    else if ((int)blockIdx.x < n_isig + spec.L)
        noise_spectrum(s1, K, blockIdx.x - n_isig, spec, w, R);
    else
        noise_peak(s1, K, peak, w);
}

// Whether the transforms are accurate enough for these inputs: *direct = 0, else 1 and the call takes the
// direct correlation.  The rounding of a transform spreads over its whole image,
// about 2^-24 of the image's rms level, while the direct sums round relative to what a pixel's own
// window holds: where sigma_eff differs much over the grid, or a region is masked, a faint pixel
// would lose accuracy (sigma rising by 1e6 across the grid: 0.1 % rms; a masked corner: noise of 1e-7 of
// the level where there is none).  So the faintest pixel's level is compared with the rms: level^2 =
// sum_q s[q]^2 isig[v + q - o]^2, the variance of y[v], over the taps within kLevelBox of the peak.
// The direct sums round the more the longer they are.  Measured on the faintest pixels of a grid whose
// halves differ in sigma (F = 128, first plane; rms / faintest level: direct / transforms, 1e-7): K = 15,
// 1.8: 1.0 / 0.8, 2.8: 1.0 / 0.9, 5.2: 1.0 / 1.3; K = 21, 4.0: 2.3 / 2.0, 5.2: 2.2 / 2.2; K = 33, 5.2: 3.6 / 2.1, 10:
// 3.6 / 4.2; K = 64, 9.2: 2.6 / 1.4 (the second plane equal there), 18: 2.5 / 2.7.  Hence K / 8, at least
// 2.5: an even grid has 1.8 (a quarter of the PSF at its corners), a 300-epoch quasar field 3.2.
constexpr int kLevelBox = 6, kLevelBlocks = 152;
constexpr float kLevelRange = 1e12f;  // 1 / sigma_eff and the PSF's norm within 1e-12 .. 1e12: no overflow
struct LevelPart {
    float least, most;  // level^2, isig
    double power;       // sum of isig^2
};
// Block b of nb.
__device__ __noinline__ void noise_level(const float *__restrict__ isig, const float *__restrict__ s1, int F, int K, int L,
                                         const NoisePeak *__restrict__ peak, LevelPart *part, int *done,
                                         int *__restrict__ direct, int b, int nb) {
    __shared__ LevelPart s_part[8];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, o = K / 2;
    const int cy = peak->qy - kLevelBox, cx = peak->qx - kLevelBox;
    LevelPart p{INFINITY, 0.f, 0.0};
    // four lanes a pixel, each a quarter of the box's rows
    for (int w = b * 256 + (int)threadIdx.x - lane; w < 4 * F * F; w += nb * 256) {
        const int u = (w + lane) >> 2, y = u / F, x = u - y * F;
        float lv = 0.f;
#pragma unroll
        for (int a0 = 0; a0 <= 2 * kLevelBox; a0 += 4) {
            const int a = a0 + (lane & 3), qy = cy + a, gy = y + qy - o;
            if (a > 2 * kLevelBox || u >= F * F || qy < 0 || qy >= K || gy < 0 || gy >= F) continue;
            float v[2 * kLevelBox + 1];
#pragma unroll
            for (int c = 0; c <= 2 * kLevelBox; ++c) {  // a row's loads together
                const int qx = cx + c, gx = x + qx - o;
                const bool in = qx >= 0 && qx < K && gx >= 0 && gx < F;
                v[c] = in ? __ldg(s1 + qy * K + qx) * __ldg(isig + gy * F + gx) : 0.f;
            }
#pragma unroll
            for (int c = 0; c <= 2 * kLevelBox; ++c) lv = fmaf(v[c], v[c], lv);
        }
        lv += __shfl_xor_sync(0xffffffffu, lv, 1);
        lv += __shfl_xor_sync(0xffffffffu, lv, 2);
        if (u < F * F && (lane & 3) == 0) {
            const float i = isig[u];
            p.least = fminf(p.least, lv);
            p.most = fmaxf(p.most, i);
            p.power += (double)i * (double)i;
        }
    }
    auto join = [](LevelPart a, LevelPart b) { return LevelPart{fminf(a.least, b.least), fmaxf(a.most, b.most), a.power + b.power}; };
    auto warp_join = [&](LevelPart a) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1)
            a = join(a, LevelPart{__shfl_down_sync(0xffffffffu, a.least, d), __shfl_down_sync(0xffffffffu, a.most, d),
                                  __shfl_down_sync(0xffffffffu, a.power, d)});
        return a;
    };
    p = warp_join(p);
    if (lane == 0) s_part[warp] = p;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) p = join(p, s_part[k]);
        part[b] = p;
        __threadfence();
        s_last = atomicAdd(done, 1) == nb - 1;
    }
    __syncthreads();
    if (!s_last || warp != 0) return;
    __threadfence();
    LevelPart t{INFINITY, 0.f, 0.0};
    for (int k = lane; k < nb; k += 32) t = join(t, part[k]);
    t = warp_join(t);
    if (lane == 0) {
        const float norm = (float)sqrt(peak->norm2);
        // the rms over a transform's L x L points; of one tile of several, at most the brightest pixel's
        const float rms = norm * fminf(t.most, (float)sqrt(t.power / ((double)L * (double)L)));
        const float limit = fmaxf(2.5f, (float)K / 8.f);
        const bool even = sqrtf(t.least) * limit >= rms;  // false for a NaN
        const bool range = t.most <= kLevelRange && t.most >= 1.f / kLevelRange && norm <= kLevelRange && norm >= 1.f / kLevelRange;
        *direct = even && range ? 0 : 1;
    }
}

template <typename Int>
__global__ void __launch_bounds__(256) noise_draw_kernel(const float *__restrict__ isig, int F, uint64_t seed,
                                                         long long r0, int B, float *__restrict__ x) {
    noise_draw<Int>(isig, F, seed, r0, B, x, blockIdx.x, gridDim.x);
}

// The first batch's draw where the transforms may run: blocks [0, n_level) look at the level, beside it.
template <typename Int>
__global__ void __launch_bounds__(256)
noise_first_draw_kernel(const float *__restrict__ isig, int F, uint64_t seed, int B, float *__restrict__ x, int n_level,
                        const float *__restrict__ s1, int K, int L, const NoisePeak *__restrict__ peak, LevelPart *part,
                        int *done, int *__restrict__ direct) {
    if ((int)blockIdx.x < n_level) noise_level(isig, s1, F, K, L, peak, part, done, direct, blockIdx.x, n_level);
    else noise_draw<Int>(isig, F, seed, 0, B, x, blockIdx.x - n_level, gridDim.x - n_level);
}

// Whether S_1^T runs as transforms (noise_fft.cu) rather than as the direct correlation, by cost per
// realisation: the multiply-adds of the direct form (its whole 32 x 128 tiles, kernel rows padded to
// 4) against the n^2 L^2 points of the transforms.  Measured per 1000 realisations (direct / transforms,
// ms): equal at about 75 multiply-adds per point (F = 64, K = 5: 0.041 / 0.039 at 63; F = 144, K = 5:
// 0.193 / 0.203 at 64; F = 90, K = 7: 0.068 / 0.076 at 75; F = 128, K = 9: 0.139 / 0.139 at 85); beyond,
// F = 128, K = 15: 0.214 / 0.141, K = 64: 2.41 / 0.174; F = 200, K = 64 (2 x 2 tiles): 8.2 / 0.78.
constexpr double kDirectPerPoint = 75.0;
bool noise_uses_fft(int F, int K, int optin, NoiseFft *plan) {
    if (!noise_fft_plan(F, K, optin, plan)) return false;
    const double tiles = (double)((F + kCorrTX - 1) / kCorrTX) * ((F + kCorrTY - 1) / kCorrTY);
    const double direct = tiles * kCorrTX * kCorrTY * K * ((K + 3) & ~3);
    return direct > kDirectPerPoint * (double)plan->n * plan->n * plan->L * plan->L;
}

// The call's workspace in one allocation: blocks are reserved, then placed (each allocation and its
// release cost about 50 us of host time, eleven of them a quarter of a call).
struct Workspace {
    struct Block {
        void **p;
        size_t off;
    };
    std::vector<Block> blocks;
    size_t bytes = 0;
    void *base = nullptr;
    ~Workspace() {
        if (base) cudaFree(base);
    }
    template <class T> void reserve(T **p, size_t count) {
        *p = nullptr;
        blocks.push_back({reinterpret_cast<void **>(p), bytes});
        bytes += (count * sizeof(T) + 255) / 256 * 256;
    }
    sr_status place() {
        const cudaError_t e = cudaMalloc(&base, bytes);
        if (e != cudaSuccess) {
            cudaGetLastError();
            base = nullptr;
            set_error("sr_noise_weights: cudaMalloc of %zu bytes failed: %s", bytes, cudaGetErrorString(e));
            return SR_ERR_OOM;
        }
        for (const Block &b : blocks) *b.p = static_cast<char *>(base) + b.off;
        return SR_OK;
    }
};

}  // namespace
}  // namespace sr

using namespace sr;

extern "C" sr_status sr_noise_weights(int N, int f, int K, int J, int E, const float *sigma_dev,
                                      const float *s1_dev, int n_real, uint64_t seed, float *W_host,
                                      float *W_map_dev, sr_noise_timing *timing, void *cuda_stream) {
    if (!sigma_dev || !s1_dev || (!W_host && !W_map_dev)) {
        set_error("sr_noise_weights: sigma, s1 and at least one output are required");
        return SR_ERR_ARG;
    }
    if (N < 1 || f < 1 || K < 1 || E < 1 || J < 2 || n_real < 2 || (long long)f * N > 65535) {
        set_error("sr_noise_weights: need N, f, K, E >= 1, J >= 2, n_real >= 2 and f N <= 65535");
        return SR_ERR_SHAPE;
    }
    const int F = f * N;
    if (J > 31 || 2LL * (1LL << (J - 2)) > F - 1) {
        set_error("sr_noise_weights: the starlet needs 2 * 2^(J-2) <= F - 1 (F = %d, J = %d)", F, J);
        return SR_ERR_SHAPE;
    }
    const int KP = (K + 3) & ~3;
    int dev = 0, sms = 0, optin = 0, per_sm = 0;
    SR_CUDA(cudaGetDevice(&dev));
    SR_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    SR_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    SR_CUDA(cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
    // kernel rows per chunk (at least RY; rows beyond K are zero): the largest that lets
    // kCorrMinBlocks blocks share an SM (1 KB reserved per block), else the largest that fits one
    int KC = 0;
    for (int kc : {64, 32, 16, 8})
        if (kCorrMinBlocks * (corr_smem_bytes(KP, std::max(std::min(kc, K), kCorrRY)) + 1024) <= (size_t)per_sm) {
            KC = std::max(std::min(kc, K), kCorrRY);
            break;
        }
    if (!KC)
        for (int kc : {32, 16, 8})
            if (corr_smem_bytes(KP, std::max(std::min(kc, K), kCorrRY)) <= (size_t)optin) {
                KC = std::max(std::min(kc, K), kCorrRY);
                break;
            }
    if (!KC) {
        set_error("sr_noise_weights: PSF size K = %d needs more shared memory than a block has", K);
        return SR_ERR_UNSUPPORTED;
    }
    // the transform form of the correlation where it is the cheaper one
    NoiseFft fft;
    const bool use_fft = noise_uses_fft(F, K, optin, &fft);
    const size_t corr_smem = corr_smem_bytes(KP, KC);
    SR_CUDA(cudaFuncSetAttribute(noise_corr_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)corr_smem));
    int occ = 0;
    SR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, noise_corr_kernel, kCorrThreads, corr_smem));
    occ = std::max(occ, 1);

    // batch: whole waves of correlation blocks, two F x F float buffers per realisation within 64 MB
    const long long FF = (long long)F * F;
    const int tiles_x = (F + kCorrTX - 1) / kCorrTX, tiles_y = (F + kCorrTY - 1) / kCorrTY;
    const long long bmax = std::max(1LL, (64LL << 20) / (2 * 4 * FF));
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);

    sr_status rc;
    NoiseSpec spec;
    long long tiles = (long long)tiles_x * tiles_y, resident = (long long)occ * sms;
    if (use_fft) {
        int blocks = 0;
        if ((rc = noise_fft_prepare(fft, &blocks)) != SR_OK) return rc;
        tiles = (long long)fft.n * fft.n;  // per pair of realisations
        resident = 2LL * std::max(blocks, 1) * sms;
    }
    long long B = std::max(1LL, (std::max(1LL, bmax * tiles / resident) * resident) / tiles);
    B = std::min({B, bmax, (long long)n_real, 65535LL});
    if (use_fft && B < n_real && B > 1) B &= ~1LL;  // whole pairs of realisations
    // segments of the moment sums: enough threads in the column pass to fill the GPU
    const int S = (int)std::max(1LL, std::min({16LL, B, (sms * 2048LL + FF - 1) / FF}));
    const int J1 = J - 1;
    Workspace ws;
    float *isig, *xbuf, *cbuf, *wsc;
    double2 *scale_part;
    double *acc1, *acc2;
    int *flag;  // flag, direct; J1 + 1 finishing counters
    NoisePeak *peak = nullptr;
    LevelPart *level_part = nullptr;
    ws.reserve(&acc1, (size_t)S * J1 * FF);
    ws.reserve(&acc2, (size_t)S * J1 * FF);
    ws.reserve(&flag, 3 + J1);
    const size_t zeroed = ws.bytes;
    ws.reserve(&isig, FF);
    ws.reserve(&xbuf, B * FF);
    ws.reserve(&cbuf, B * FF);
    ws.reserve(&wsc, J1);
    ws.reserve(&scale_part, (size_t)J1 * kScaleBlocks);
    if (use_fft) {
        ws.reserve(&spec.S, (size_t)fft.L * fft.L);
        ws.reserve(&spec.tw, fft.L);
        ws.reserve(&peak, 1);
        ws.reserve(&level_part, kLevelBlocks);
        spec.L = fft.L;
        spec.R1 = fft.R1;
        spec.sh = fft.n == 1 ? K / 2 : 0;
        noise_fft_gain(fft, spec.gain);
    }
    if ((rc = ws.place()) != SR_OK) return rc;
    SR_CUDA(cudaMemsetAsync(ws.base, 0, zeroed, st));  // the moments, the flag and the finishing counters

    cudaEvent_t ev[5] = {};
    const bool timed = timing != nullptr;
    double t_draw = 0, t_corr = 0, t_star = 0, t_fin = 0;
    int launches = 0;
    auto destroy_events = [&]() {
        for (cudaEvent_t &e : ev)
            if (e) cudaEventDestroy(e), e = nullptr;
    };
    if (timed)
        for (cudaEvent_t &e : ev)
            if (cudaEventCreate(&e) != cudaSuccess) {
                destroy_events();
                return cuda_fail(cudaGetLastError(), "cudaEventCreate");
            }
    auto elapsed = [&](int a, int b) -> double {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, ev[a], ev[b]);
        return ms;
    };

    const int n_isig = (int)std::min<long long>(((long long)N * N + 31) / 32, sms * 8LL);
    noise_setup_kernel<<<n_isig + spec.L + (use_fft ? 1 : 0), 32 * kIsigWarps, 0, st>>>(sigma_dev, s1_dev, N, f, E, K,
                                                                                        n_isig, isig, flag, spec, peak);
    ++launches;
    const int n_level = (int)std::min<long long>((4 * FF + 255) / 256, kLevelBlocks);
    // The transforms' first batch runs before the host knows whether they are to be used: asking first would
    // leave the GPU idle for the answer (a call of 400 us took 445).
    bool fft_now = use_fft;
    int found[2] = {0, 0};  // bad inputs; use the direct form
    auto read_found = [&]() -> cudaError_t {
        cudaError_t e = cudaMemcpyAsync(found, flag, sizeof found, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        return e;
    };
    auto start_over = [&]() -> cudaError_t {  // what the transforms' batches left
        fft_now = false;
        launches = 1;
        return cudaMemsetAsync(ws.base, 0, zeroed, st);
    };
    cudaError_t e = cudaSuccess;
    for (;;) {
        for (long long r0 = 0; r0 < n_real; r0 += B) {
            if (fft_now && r0 == B) {
                e = read_found();
                if (e == cudaSuccess && found[1]) {
                    e = start_over();
                    r0 = 0;
                }
                if (e != cudaSuccess) break;
            }
            const int Bb = (int)std::min(B, (long long)n_real - r0);
            const int *skip = fft_now ? flag + 1 : nullptr;
            if (timed) cudaEventRecord(ev[0], st);
            const long long nblk = ((r0 + Bb) * FF - 1) / 4 - (r0 * FF) / 4 + 1;
            const int gd = (int)std::min<long long>((nblk + 255) / 256, sms * 16LL);
            const bool small = Bb * FF < (1LL << 30);
            if (fft_now && r0 == 0) {
                int *done = flag + 2 + J1;
                if (small)
                    noise_first_draw_kernel<int><<<n_level + gd, 256, 0, st>>>(isig, F, seed, Bb, xbuf, n_level, s1_dev, K,
                                                                               spec.L, peak, level_part, done, flag + 1);
                else
                    noise_first_draw_kernel<long long><<<n_level + gd, 256, 0, st>>>(isig, F, seed, Bb, xbuf, n_level, s1_dev,
                                                                                     K, spec.L, peak, level_part, done, flag + 1);
            } else if (small) {
                noise_draw_kernel<int><<<gd, 256, 0, st>>>(isig, F, seed, r0, Bb, xbuf);
            } else {
                noise_draw_kernel<long long><<<gd, 256, 0, st>>>(isig, F, seed, r0, Bb, xbuf);
            }
            if (timed) cudaEventRecord(ev[1], st);
            if (fft_now) {
                if ((rc = launch_noise_fft(fft, xbuf, spec.S, spec.tw, F, K, Bb, sms, skip, cbuf, st)) != SR_OK) {
                    destroy_events();
                    return rc;
                }
            } else {
                noise_corr_kernel<<<dim3(tiles_x, tiles_y, Bb), kCorrThreads, corr_smem, st>>>(xbuf, s1_dev, F, K, KP, KC,
                                                                                               cbuf);
            }
            if (timed) cudaEventRecord(ev[2], st);
            const long long total = Bb * FF;
            const int Sb = std::min(S, Bb);
            for (int j = 0; j < J1; ++j) {
                noise_row_kernel<<<(int)std::min<long long>((total + 255) / 256, sms * 16LL), 256, 0, st>>>(
                    cbuf, xbuf, F, 1 << j, total, skip);
                noise_col_stats_kernel<<<dim3((unsigned)((FF + 255) / 256), Sb), 256, 0, st>>>(
                    cbuf, xbuf, F, 1 << j, Bb, Sb, J1, j, acc1, acc2);
            }
            launches += 2 + 2 * J1;
            if (timed) {
                cudaEventRecord(ev[3], st);
                if ((e = cudaEventSynchronize(ev[3])) != cudaSuccess) break;
                t_draw += elapsed(0, 1);
                t_corr += elapsed(1, 2);
                t_star += elapsed(2, 3);
            }
        }
        if (e != cudaSuccess) {
            destroy_events();
            return cuda_fail(e, "noise propagation batch");
        }
        if (timed) cudaEventRecord(ev[0], st);
        if (W_map_dev) {
            const long long per = (long long)J1 * FF;
            noise_map_kernel<<<(unsigned)((per + 255) / 256), 256, 0, st>>>(acc1, acc2, per, S, n_real, W_map_dev);
            ++launches;
        }
        noise_scale_kernel<<<dim3(kScaleBlocks, J1), kScaleThreads, 0, st>>>(acc1, acc2, FF, J1, S, n_real, scale_part,
                                                                               flag + 2, wsc);
        ++launches;
        if (timed) cudaEventRecord(ev[4], st);
        e = cudaGetLastError();
        if (e != cudaSuccess) {
            destroy_events();
            return cuda_fail(e, "noise propagation kernels");
        }
        if (W_host) e = cudaMemcpyAsync(W_host, wsc, sizeof(float) * J1, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = fft_now || !use_fft ? read_found() : cudaStreamSynchronize(st);
        if (e == cudaSuccess && fft_now && found[1]) {  // one batch in all
            e = start_over();
            if (e == cudaSuccess) continue;
        }
        if (e != cudaSuccess) {
            destroy_events();
            return cuda_fail(e, "sr_noise_weights");
        }
        break;
    }
    const int hflag = found[0];
    if (timed) {
        t_fin = elapsed(0, 4);
        timing->draw_ms = t_draw;
        timing->corr_ms = t_corr;
        timing->starlet_ms = t_star;
        timing->final_ms = t_fin;
        timing->launches = launches;
        timing->batch = (int)B;
        destroy_events();
    }
    if (hflag) {
        set_error("sr_noise_weights: %s", (hflag & 1) ? "sigma holds a NaN or a value <= 0" : "s1 is not finite");
        return SR_ERR_NONFINITE;
    }
    return SR_OK;
}
