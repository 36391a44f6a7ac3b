// S_1^T of the noise propagation by transforms (sm_103a): the zero-padded correlation
//     y[v] = sum_q s[q] x[v + q - o]     (o = K/2; x = 0 outside the F x F grid)
// of noise.cu, evaluated with circular transforms of L x L in shared memory.
//
// Two realisations travel as the real and imaginary parts of one complex image; both are multiplied
// by the same spectrum, so nothing has to be separated between the transforms.  A realisation is cut
// into n x n output tiles of T x T:
//   n = 1   x is placed at 0 and padded with zeros, L >= F + max(o, K - 1 - o) keeps the output free
//           of wrap-around (tap q at (q - o) mod L);
//   n > 1   a tile reads the patch of T + K - 1 <= L values it needs, placed at 0 (tap q at q).
// The passes are those of fft_pair.cuh, with the last pass along y, the product and the first inverse
// pass along y in registers (one round trip through shared memory and two barriers fewer):
//   rows (2 passes over the patch rows) | columns, pass A | pass B, product, pass B inverse |
//   columns, pass A inverse | rows inverse (2 passes over the output rows).
//
// Against the direct correlation, which is bound by FP32 FMA issue at 2 K^2 flop per pixel, a pixel
// costs about 20 log2 L flop here; bound by the latency of the passes (one block of 512 threads per
// SM at L = 160): 5000 realisations at F = 128, K = 64 take 0.78 ms, the direct form 11.7 ms.
#include <math.h>

#include <algorithm>
#include <complex>
#include <mutex>

#include "common.cuh"
#include "cplx.cuh"
#include "fft_pair.cuh"
#include "noise.cuh"
#include "once.cuh"

namespace sr {
namespace {

#define SR_NF_SIZES(X) /* multiples of 8 up to kNoiseMaxL */ \
    X(32) X(40) X(48) X(56) X(64) X(72) X(80) X(96) X(112) X(128) X(144) X(160)

constexpr int kNfThreads = 512;

template <int L>
constexpr int nf_smem() {
    return (Pr<L>::ZN + L) * (int)sizeof(float2);
}

// One item: the tile (ty, tx) of realisations 2p and 2p + 1 of the batch.
template <int L>
__global__ void __launch_bounds__(kNfThreads, 1)
noise_fft_kernel(const float *__restrict__ x, const float2 *__restrict__ S, const float2 *__restrict__ tw, int F, int K,
                 int n, int T, int B, int n_items, const int *__restrict__ skip, float *__restrict__ y) {
    if (*skip) return;
    using G = Pr<L>;
    constexpr int R1 = G::R1, R2 = G::R2, P = G::P;
    float2 *Z = pr_dyn, *TWL = Z + G::ZN;
    const int tid = threadIdx.x, nt = blockDim.x;
    load_twl<L>(TWL, tw);
    const long long FF = (long long)F * F;
    const int off = n > 1 ? K / 2 : 0;
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int p = item / (n * n), tile = item - p * n * n;
        const int vy = (tile / n) * T, vx = (tile % n) * T;
        const int ny = min(T, F - vy), nx = min(T, F - vx);           // outputs
        const int py = n > 1 ? ny + K - 1 : F, px = n > 1 ? nx + K - 1 : F;  // inputs
        const float *xa = x + 2LL * p * FF;
        const bool has1 = 2 * p + 1 < B;
        const float inv_px = 1.f / (float)px;
        for (int t = tid; t < py * px; t += nt) {
            const int r = fdivq(t, inv_px), c = t - r * px;
            const int gy = vy - off + r, gx = vx - off + c;
            float2 v = make_float2(0.f, 0.f);
            if (gy >= 0 && gy < F && gx >= 0 && gx < F) {
                const long long u = (long long)gy * F + gx;
                v = make_float2(__ldg(xa + u), has1 ? __ldg(xa + FF + u) : 0.f);
            }
            Z[r * P + pcol<L>(c)] = v;
        }
        __syncthreads();
        rows_fwd<L>(Z, 1, py, px, TWL);
        for (int t = tid; t < R2 * L; t += nt) {  // columns, pass A
            const int c = t % L, n2 = t / L;
            float2 *z = Z + pcol<L>(c) + n2 * P;
            float2 v[R1];
#pragma unroll
            for (int n1 = 0; n1 < R1; ++n1) v[n1] = n2 + R2 * n1 < py ? z[R2 * n1 * P] : make_float2(0.f, 0.f);
            dft<R1, false>(v);
#pragma unroll
            for (int k1 = 0; k1 < R1; ++k1) z[R2 * k1 * P] = k1 == 0 ? v[0] : cmul(v[k1], TWL[k1 * R2 + n2]);
        }
        __syncthreads();
        for (int t = tid; t < R1 * L; t += nt) {  // columns, pass B, the product, pass B inverse
            const int c = t % L, k1 = t / L;
            float2 *z = Z + pcol<L>(c) + R2 * k1 * P;
            const float2 *sp = S + (long long)R2 * k1 * L + c;
            float2 v[R2], sv[R2];
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2) sv[k2] = __ldg(sp + k2 * L);
#pragma unroll
            for (int n2 = 0; n2 < R2; ++n2) v[n2] = z[n2 * P];
            dft<R2, false>(v);
#pragma unroll
            for (int k2 = 0; k2 < R2; ++k2) v[k2] = cmul(v[k2], sv[k2]);
            dft<R2, true>(v);
#pragma unroll
            for (int n2 = 0; n2 < R2; ++n2) z[n2 * P] = n2 == 0 ? v[0] : cmulc(v[n2], TWL[k1 * R2 + n2]);
        }
        __syncthreads();
        for (int t = tid; t < R2 * L; t += nt) {  // columns, pass A inverse
            const int c = t % L, n2 = t / L;
            float2 *z = Z + pcol<L>(c) + n2 * P;
            float2 v[R1];
#pragma unroll
            for (int k1 = 0; k1 < R1; ++k1) v[k1] = z[R2 * k1 * P];
            dft<R1, true>(v);
#pragma unroll
            for (int n1 = 0; n1 < R1; ++n1)
                if (n2 + R2 * n1 < ny) z[R2 * n1 * P] = v[n1];
        }
        __syncthreads();
        rows_inv<L>(Z, 1, ny, nx, TWL);
        float *ya = y + 2LL * p * FF;
        const float inv_nx = 1.f / (float)nx;
        for (int t = tid; t < ny * nx; t += nt) {
            const int r = fdivq(t, inv_nx), c = t - r * nx;
            const float2 v = Z[r * P + pcol<L>(c)];
            const long long u = (long long)(vy + r) * F + vx + c;
            ya[u] = v.x;
            if (has1) ya[FF + u] = v.y;
        }
        __syncthreads();
    }
}

// The block size with the most threads resident per SM (ties to the smaller one: independent blocks
// cover each other's barriers), and its resident blocks.
template <typename Kern>
sr_status nf_block(Kern kernel, int smem, int *threads, int *occ) {
    SR_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    *threads = 0;
    *occ = 0;
    for (int t : {kNfThreads, kNfThreads / 2, kNfThreads / 4}) {
        int o = 0;
        SR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kernel, t, smem));
        if (o >= 1 && o * t >= *threads * *occ) {
            *threads = t;
            *occ = o;
        }
    }
    return SR_OK;
}

// the DFT twiddles of this translation unit, once per device
sr_status nf_tables() {
    static OncePerDevice once;
    return once.run([]() -> sr_status {
        SR_CUDA(pr_fill_dtw());
        return SR_OK;
    });
}

// The in-register DFTs of fft_pair.cuh (dft<R, false>) in FP64 with the same FP32 constants: v[k] in,
// X[k] out.
using cd = std::complex<double>;
cd rounded_root(int m, int R) {  // exp(-2 pi i m / R) as the kernels hold it
    if (4 * m % R == 0) {
        const cd quarter[4] = {cd(1, 0), cd(0, -1), cd(-1, 0), cd(0, 1)};
        return quarter[4 * m / R % 4];
    }
    const double a = -2.0 * M_PI * (double)m / (double)R;
    return cd((float)cos(a), (float)sin(a));
}
void rounded_dft(int R, cd *v) {
    int P = 0;
    switch (R) {
        case 6: case 8: case 10: P = 2; break;
        case 9: P = 3; break;
        case 16: P = 4; break;
        default: break;
    }
    if (P == 0) {  // 2 .. 5 and 7 points: their sums over v with FP32 cosines and sines
        cd X[8];
        for (int k = 0; k < R; ++k) {
            X[k] = 0.0;
            for (int j = 0; j < R; ++j) X[k] += v[j] * rounded_root(j * k % R, R);
        }
        std::copy(X, X + R, v);
        return;
    }
    const int Q = R / P;  // dft_pq
    cd a[16], t[16];
    for (int n2 = 0; n2 < Q; ++n2) {
        for (int n1 = 0; n1 < P; ++n1) t[n1] = v[Q * n1 + n2];
        rounded_dft(P, t);
        for (int k1 = 0; k1 < P; ++k1) a[k1 * Q + n2] = t[k1] * rounded_root(n2 * k1, R);
    }
    for (int k1 = 0; k1 < P; ++k1) {
        for (int n2 = 0; n2 < Q; ++n2) t[n2] = a[k1 * Q + n2];
        rounded_dft(Q, t);
        for (int k2 = 0; k2 < Q; ++k2) v[k1 + P * k2] = t[k2];
    }
}

}  // namespace

// A unit wave of frequency k goes in, and what comes out at k is the mean of the rounded roots over the
// exact ones; the way back multiplies by the same, conjugated.  With L = R1 R2, n = n2 + R2 n1 and
// k = k1 + R1 k2 the mean factors into those of the two passes.  Without the correction the weights came
// out 7e-8 to 1.2e-7 too small at L = 48, 64, 96, 128 and 144 (a rounding of the result is 6e-8).
static void gain_of(int L, int R1, double *gain) {
    const int R2 = L / R1;
    auto exact = [](int m, int R) { return std::polar(1.0, 2.0 * M_PI * (double)(m % R) / (double)R); };  // conjugate
    auto matrix = [](int R, cd *D) {  // D[k R + n]: row k of the R-point transform
        for (int n = 0; n < R; ++n) {
            cd v[16] = {};
            v[n] = 1.0;
            rounded_dft(R, v);
            for (int k = 0; k < R; ++k) D[k * R + n] = v[k];
        }
    };
    cd D1[16 * 16], D2[16 * 16];
    matrix(R1, D1);
    matrix(R2, D2);
    for (int k = 0; k < L; ++k) {
        const int k1 = k % R1, k2 = k / R1;
        cd a = 0.0, b = 0.0;
        for (int n1 = 0; n1 < R1; ++n1) a += D1[k1 * R1 + n1] * exact(k1 * n1, R1);
        for (int n2 = 0; n2 < R2; ++n2)
            b += D2[k2 * R2 + n2] * exact(k2 * n2, R2) * (k1 == 0 ? cd(1.0) : rounded_root(k1 * n2, L) * exact(k1 * n2, L));
        gain[k] = std::norm(a * b / (double)L);
    }
}

void noise_fft_gain(const NoiseFft &plan, double *gain) {
    static std::mutex m;
    static double table[kNoiseMaxL / 8 + 1][kNoiseMaxL];  // by L / 8; 40 us to fill a row
    static bool done[kNoiseMaxL / 8 + 1];
    const int i = plan.L / 8;
    std::lock_guard<std::mutex> lock(m);
    if (!done[i]) {
        gain_of(plan.L, plan.R1, table[i]);
        done[i] = true;
    }
    std::copy(table[i], table[i] + plan.L, gain);
}

bool noise_fft_plan(int F, int K, int smem_optin, NoiseFft *plan) {
    static const int sizes[] = {
#define SR_NF_LIST(LL) LL,
        SR_NF_SIZES(SR_NF_LIST)
#undef SR_NF_LIST
    };
    const int o = K / 2;
    double best = 0.0;
    for (int n = 1; n <= F && n <= 64; ++n) {
        const int T = (F + n - 1) / n, need = n == 1 ? F + (o > K - 1 - o ? o : K - 1 - o) : T + K - 1;
        if ((long long)T * (n - 1) >= F) continue;  // an empty last tile
        for (int L : sizes) {
            if (L < need || L < K) continue;
            int smem = 0;
            switch (L) {
#define SR_NF_SM(LL)           \
    case LL:                   \
        smem = nf_smem<LL>();  \
        break;
                SR_NF_SIZES(SR_NF_SM)
#undef SR_NF_SM
                default:
                    break;
            }
            if (smem > smem_optin) break;
            const double cost = (double)n * n * L * L;
            if (best == 0.0 || cost < best) {
                best = cost;
                plan->L = L;
                plan->R1 = pr_r1(L);
                plan->n = n;
                plan->T = T;
            }
            break;  // the smallest size that fits
        }
    }
    return best > 0.0;
}

sr_status noise_fft_prepare(const NoiseFft &plan, int *resident) {
    sr_status rc = nf_tables();
    if (rc != SR_OK) return rc;
    int threads = 0, occ = 0;
    switch (plan.L) {
#define SR_NF_OCC(LL)                                                       \
    case LL:                                                                \
        rc = nf_block(noise_fft_kernel<LL>, nf_smem<LL>(), &threads, &occ); \
        break;
        SR_NF_SIZES(SR_NF_OCC)
#undef SR_NF_OCC
        default:
            break;
    }
    *resident = occ;
    return rc;
}

sr_status launch_noise_fft(const NoiseFft &plan, const float *x, const float2 *S, const float2 *tw, int F, int K, int B,
                           int n_sms, const int *skip, float *y, cudaStream_t st) {
    const int items = (B + 1) / 2 * plan.n * plan.n;
    int threads = 0, occ = 0;
    switch (plan.L) {
#define SR_NF_RUN(LL)                                                                                          \
    case LL: {                                                                                                 \
        const sr_status rc = nf_block(noise_fft_kernel<LL>, nf_smem<LL>(), &threads, &occ);                    \
        if (rc != SR_OK) return rc;                                                                            \
        const int grid = items < occ * n_sms ? items : occ * n_sms;                                            \
        noise_fft_kernel<LL><<<grid, threads, nf_smem<LL>(), st>>>(x, S, tw, F, K, plan.n, plan.T, B, items,   \
                                                                   skip, y);                                   \
        break;                                                                                                 \
    }
        SR_NF_SIZES(SR_NF_RUN)
#undef SR_NF_RUN
        default:
            break;
    }
    return SR_OK;
}

}  // namespace sr
