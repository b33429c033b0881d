// What a trainer-side batch still needs after the features: cepstra (the MFCC
// baseline of the paper's Table 1 is a DCT of log-mel energies), per-utterance mean
// and variance of every feature, and an ordering of utterances by length for
// padded batches (Section 2.2).
#include <cooperative_groups.h>

#include <algorithm>
#include <numeric>
#include <vector>

#include "common.cuh"
#include "fft_pair.cuh"

namespace {

// c_i = s_i sum_m x[m] cos(pi i (m + 1/2) / M), s_0 = sqrt(1/M), s_i = sqrt(2/M): orthonormal DCT-II
//
// A small matrix product, bound by reading the features once (80 bands: 320 bytes and 1040
// multiply-adds a frame) as long as they are not read again for every coefficient: a CTA
// stages a tile of 128 frames in shared memory and each thread carries eight coefficients of two frames, the
// basis arriving as 128-bit broadcasts.  The features are copied asynchronously while the basis is worked out, and read
// back four bands at a time.  205 k frames, 80 bands, 13 coefficients (the bytes take 12 us), and what else it takes to make
// them from the waveform: 318 us in all with loads through registers and one band at a time, 293.
constexpr int MFCC_THREADS = 128, MFCC_FT = 128, MFCC_CB = 16;   // frames per tile, coefficients per round
// Rows of a staged frame: an odd number of 16-byte words, so that both copies of whole words and the reads of 32 frames'
// words are free of bank conflicts.
__host__ __device__ constexpr int mfcc_ld(int M) { return 4 * (((M + 3) >> 2) | 1); }
__host__ __device__ constexpr size_t mfcc_smem(int M) {
    return sizeof(float) * ((size_t)MFCC_FT * mfcc_ld(M) + MFCC_CB * ((M + 3) & ~3) + MFCC_FT * (MFCC_CB + 1) + 4);
}
__global__ void __launch_bounds__(MFCC_THREADS)
mfcc_kernel(const float *__restrict__ feats, const int *__restrict__ counts, int M, int n_cep,
            int T_max, float pad_v, float *__restrict__ out) {
    extern __shared__ __align__(16) float sm[];
    float *basis = sm;                               // [M][MFCC_CB]
    const int M4 = (M + 3) & ~3;                     // bands, and zeros up to whole words
    float *xs = basis + MFCC_CB * M4;                // [MFCC_FT][mfcc_ld(M)]
    const int utt = blockIdx.y, tid = threadIdx.x, ld = mfcc_ld(M);
    float *os = xs + MFCC_FT * ld;                   // [MFCC_FT][MFCC_CB + 1]
    const int t0 = blockIdx.x * MFCC_FT;
    const int rows = min(MFCC_FT, T_max - t0);
    const int T = min(max(counts[utt], 0), T_max);
    const int nf = min(rows, T - t0);                // frames of this tile that hold features
    float *o = out + ((int64_t)utt * T_max + t0) * n_cep;
    for (int i = max(nf, 0) * n_cep + tid; i < rows * n_cep; i += MFCC_THREADS) o[i] = pad_v;
    if (nf <= 0) return;
    const float *x = feats + ((int64_t)utt * T_max + t0) * M;
    if ((M & 3) == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0) {
        const int m4 = M >> 2, step_f = MFCC_THREADS / m4, step_m = MFCC_THREADS - step_f * m4;
        int f = tid / m4, m = tid - f * m4;
        const float *src = x + 4 * tid;
        for (int i = tid; i < nf * m4; i += MFCC_THREADS, src += 4 * MFCC_THREADS) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                             (unsigned)__cvta_generic_to_shared(xs + f * ld + 4 * m)), "l"(src) : "memory");
            f += step_f;
            m += step_m;
            if (m >= m4) {
                m -= m4;
                ++f;
            }
        }
    } else {
        for (int i = tid; i < MFCC_FT * (M4 - M); i += MFCC_THREADS) xs[i / (M4 - M) * ld + M + i % (M4 - M)] = 0.f;
        for (int i = tid; i < nf * M; i += MFCC_THREADS) {
            const int f = i / M;
            xs[i + f * (ld - M)] = __ldg(x + i);
        }
    }
    const int f0 = tid & 63, half = tid >> 6;
    for (int c0 = 0; c0 < n_cep; c0 += MFCC_CB) {
        const int nc = min(MFCC_CB, n_cep - c0);
        // A thread's coefficient c is always the same; k = c (2 m + 1) mod 4 M, the angle in units of
        // pi / 2M, goes from one of its bands to the next.
        const int c = c0 + tid % MFCC_CB, step = 2 * c * (MFCC_THREADS / MFCC_CB) % (4 * M);
        const float s = c >= n_cep ? 0.f : c == 0 ? rsqrtf((float)M) : sqrtf(2.f / (float)M);
        const float unit = 1.f / (float)(2 * M), rest = fmaf(-unit, (float)(2 * M), 1.f) * unit;   // 1 / 2M in two parts
        int k = c * (2 * (tid / MFCC_CB) + 1) % (4 * M);
        for (int i = tid; i < MFCC_CB * M4; i += MFCC_THREADS) {
            basis[i] = i < MFCC_CB * M ? s * cospif(fmaf((float)k, unit, (float)k * rest)) : 0.f;
            k += step;
            if (k >= 4 * M) k -= 4 * M;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        // pairs of coefficients, as the basis is read
        fftpair::u64 a[4], b[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) a[c] = b[c] = 0;
        const float *x0 = xs + f0 * ld, *x1 = x0 + 64 * ld, *bz = basis + 8 * half;
#pragma unroll 2
        for (int m = 0; m < M4; m += 4) {
            const float4 p0 = *reinterpret_cast<const float4 *>(x0 + m), p1 = *reinterpret_cast<const float4 *>(x1 + m);
            const float e0[4] = {p0.x, p0.y, p0.z, p0.w}, e1[4] = {p1.x, p1.y, p1.z, p1.w};
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                const fftpair::u64 u = fftpair::both(e0[d]), v = fftpair::both(e1[d]);
                const ulonglong2 p = *reinterpret_cast<const ulonglong2 *>(bz + MFCC_CB * (m + d));
                const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(bz + MFCC_CB * (m + d) + 4);
                const fftpair::u64 w[4] = {p.x, p.y, q.x, q.y};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    a[c] = fftpair::fma2(u, w[c], a[c]);
                    b[c] = fftpair::fma2(v, w[c], b[c]);
                }
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float2 ua = fftpair::unpack(a[c]), ub = fftpair::unpack(b[c]);
            float *oa = os + f0 * (MFCC_CB + 1) + 8 * half + 2 * c, *ob = oa + 64 * (MFCC_CB + 1);
            oa[0] = ua.x;
            oa[1] = ua.y;
            ob[0] = ub.x;
            ob[1] = ub.y;
        }
        __syncthreads();
        const int step_f = MFCC_THREADS / nc, step_c = MFCC_THREADS - step_f * nc;
        int f = tid / nc, co = tid - f * nc;
#pragma unroll 4
        for (int i = tid; i < nf * nc; i += MFCC_THREADS) {
            o[f * n_cep + c0 + co] = os[f * (MFCC_CB + 1) + co];
            f += step_f;
            co += step_c;
            if (co >= nc) {
                co -= nc;
                ++f;
            }
        }
        __syncthreads();       // basis and the output tile are rewritten by the next round
    }
}

// Mean and variance: a pass over the features, bound by reading them.  A cluster of eight CTAs
// shares an utterance, so that a batch of a hundred utterances fills the device (one CTA per
// utterance left 5 of 6 warps' worth of loads unissued: 441 us for 128 utterances of 2-30 s
// with 80 features, 66 MB; now 18.5 while they are in L2 and 25 from memory).  Every thread keeps
// VEC columns and strides over the frames, eight loads in flight, the CTA adds its threads, and
// the first CTA adds the eight through distributed shared memory: no workspace, no atomics, the
// order of the additions is fixed.  Sums in double, so 6000 frames lose nothing.
constexpr int MV_CLUSTER = 8, MV_THREADS = 256;
template <int VEC>
__global__ void __cluster_dims__(MV_CLUSTER, 1, 1) __launch_bounds__(MV_THREADS)
mean_var_kernel(const float *__restrict__ feats, const int *__restrict__ counts, int D, int T_max,
                float *__restrict__ mean, float *__restrict__ var) {
    constexpr int COLS = VEC * MV_THREADS;           // columns per round
    __shared__ double s1[COLS], s2[COLS];
    const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int utt = blockIdx.y, rank = blockIdx.x, tid = threadIdx.x;
    const int T = min(max(counts[utt], 0), T_max);
    for (int d0 = 0; d0 < D; d0 += COLS) {
        const int cols = min(COLS, D - d0), groups = cols / VEC;
        const int slices = MV_THREADS / groups;      // frames the CTA reads side by side
        const int slice = tid / groups, g = tid - slice * groups;
        double a[VEC], b[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) a[v] = b[v] = 0.0;
        if (slice < slices) {
            const float *x = feats + (int64_t)utt * T_max * D + d0 + g * VEC;
#pragma unroll 8
            for (int t = rank * slices + slice; t < T; t += MV_CLUSTER * slices) {
                float z[VEC];
                if constexpr (VEC == 4) {
                    const float4 q = __ldg(reinterpret_cast<const float4 *>(x + (int64_t)t * D));
                    z[0] = q.x;
                    z[1] = q.y;
                    z[2] = q.z;
                    z[3] = q.w;
                } else {
                    z[0] = __ldg(x + (int64_t)t * D);
                }
#pragma unroll
                for (int v = 0; v < VEC; ++v) {
                    const double y = z[v];
                    a[v] += y;
                    b[v] = fma(y, y, b[v]);
                }
            }
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                s1[slice * cols + g * VEC + v] = a[v];
                s2[slice * cols + g * VEC + v] = b[v];
            }
        }
        __syncthreads();
        for (int d = tid; d < cols; d += MV_THREADS) {          // column d is touched by this thread alone
            for (int j = 1; j < slices; ++j) {
                s1[d] += s1[j * cols + d];
                s2[d] += s2[j * cols + d];
            }
        }
        cluster.sync();
        if (rank == 0) {
            for (int d = tid; d < cols; d += MV_THREADS) {
                double p = 0.0, q = 0.0;
#pragma unroll
                for (int c = 0; c < MV_CLUSTER; ++c) {
                    p += *cluster.map_shared_rank(&s1[d], c);
                    q += *cluster.map_shared_rank(&s2[d], c);
                }
                const double mu = T > 0 ? p / T : 0.0;
                const double vv = T > 0 ? q / T - mu * mu : 0.0;
                mean[(int64_t)utt * D + d0 + d] = (float)mu;
                var[(int64_t)utt * D + d0 + d] = (float)(vv > 0.0 ? vv : 0.0);
            }
        }
        cluster.sync();        // the sums stay in place until they have been read
    }
}

}  // namespace

extern "C" int feat_mfcc(AugCtx *ctx, const float *feats_dev, const int *counts_dev, int B, int T_max,
                         int n_cep, float *mfcc_dev) {
    if (!ctx || B < 0) return AUG_EINVAL;
    if (B > ctx->cfg.max_batch) return AUG_ECAP;
    if (B == 0) return AUG_OK;
    const int M = ctx->cfg.n_mel;
    if (!feats_dev || !counts_dev || !mfcc_dev || T_max <= 0 || n_cep < 1 || n_cep > M) return AUG_EINVAL;
    if (smem_opt_in<mfcc_kernel>(ctx->device) != AUG_OK) return AUG_ECUDA;
    dim3 grid((T_max + MFCC_FT - 1) / MFCC_FT, B);
    mfcc_kernel<<<grid, MFCC_THREADS, mfcc_smem(M), ctx->stream>>>(feats_dev, counts_dev, M, n_cep, T_max,
                                                  ctx->cfg.pad_value, mfcc_dev);
    AUG_CUDA_OK(cudaGetLastError());
    ctx->launches++;
    return AUG_OK;
}

extern "C" int feat_mean_var(AugCtx *ctx, const float *feats_dev, const int *counts_dev, int B,
                             int T_max, int D, float *mean_dev, float *var_dev) {
    if (!ctx || B < 0) return AUG_EINVAL;
    if (B > ctx->cfg.max_batch) return AUG_ECAP;
    if (B == 0) return AUG_OK;
    if (!feats_dev || !counts_dev || !mean_dev || !var_dev || T_max <= 0 || D < 1) return AUG_EINVAL;
    // four columns a thread where every row starts on a 16-byte boundary
    const bool vec = (D & 3) == 0 && (reinterpret_cast<uintptr_t>(feats_dev) & 15) == 0;
    auto kern = vec ? mean_var_kernel<4> : mean_var_kernel<1>;
    kern<<<dim3(MV_CLUSTER, B), MV_THREADS, 0, ctx->stream>>>(feats_dev, counts_dev, D, T_max, mean_dev, var_dev);
    AUG_CUDA_OK(cudaGetLastError());
    ctx->launches++;
    return AUG_OK;
}

extern "C" int aug_bucket_by_length(const int *lengths_host, int B, int batch, int *perm_host,
                                    int *batch_max_host) {
    if (B < 0 || batch < 1 || (B > 0 && (!lengths_host || !perm_host))) return AUG_EINVAL;
    std::vector<int> idx(B);
    std::iota(idx.begin(), idx.end(), 0);
    std::stable_sort(idx.begin(), idx.end(),
                     [&](int a, int b) { return lengths_host[a] < lengths_host[b]; });
    for (int i = 0; i < B; ++i) perm_host[i] = idx[i];
    if (batch_max_host)
        for (int g = 0; g * batch < B; ++g) {
            const int last = std::min(B, (g + 1) * batch) - 1;     // longest of a sorted group
            batch_max_host[g] = lengths_host[idx[last]];
        }
    return AUG_OK;
}
