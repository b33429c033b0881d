// Internal declarations shared by the translation units of libaugb200.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/aug_b200.h"

namespace aug {

constexpr int CONV_TAPS = 8192;         // taps of a partition: half a transform of the convolution
constexpr int CONV_BINS = 8192;         // complex numbers of a stored spectrum
// Counters of the convolution: the batch's largest response length (long-response contexts), units of
// work listed for the two routes (sums, blocks with copies, other ones), units drawn from the lists.
enum Counter { LEFF_ALL, LIST_FUSED, LIST_STORED = LIST_FUSED + 3, DRAWN_FUSED = LIST_STORED + 3, DRAWN_SPECTRA,
               DRAWN_STORED, N_COUNTERS };
constexpr int PARK_SLOTS = 320;     // parking slots of the fused convolution = most CTAs it runs with
constexpr int PLAN_BYTES = 96;      // per utterance, see conv.cu
constexpr int MAX_TAPS = 24576;
constexpr int MAX_ORDER = 32;
constexpr int MAX_HALF_W = 47;
constexpr int MAX_MEL = 128;
constexpr int TAP_ROWS = 13;

constexpr int EV_RING = 256;
#ifndef AUG_HOST_CHUNKS
#define AUG_HOST_CHUNKS 8
#endif
constexpr int HOST_CHUNKS = AUG_HOST_CHUNKS;   // pipeline depth of aug_pipeline_host

// How step 2 is run, fixed by the response length at aug_create:
//   ROUTE_FUSED_8192  rir_taps <= 8192: one partition of a 16384-point transform
//                     (16384 - taps + 1 outputs per block), one kernel
//   ROUTE_STORED      longer: partitions of 8192 taps, block spectra stored once and reused
enum Route { ROUTE_FUSED_8192 = 1, ROUTE_STORED = 2 };

enum Reason { R_NONE = 0, R_NSRC = 1, R_ORDER = 2, R_NOISE = 3 };

// Per-bin entry of the warped filterbank: the bin lies in edge interval `seg`
// (between edges e_seg and e_seg+1), at fraction `up` from its lower edge.
struct MelBin {
    float up;    // weight in filter seg   (rising side)
    float down;  // weight in filter seg-1 (falling side) = 1 - up
};

}  // namespace aug

struct AugCtx {
    AugConfig cfg;
    cudaStream_t stream;
    int device;
    int sm_count;          // multiprocessors of the device
    int smem_per_sm;       // shared memory of one multiprocessor, bytes
    int n_part;            // partitions of CONV_TAPS taps
    int route;             // aug::Route
    int n_bins;            // n_fft/2 + 1
    int t_cap;             // frames of an utterance of max_samples
    int64_t ws_stride;     // row stride (floats) of the y_s / v workspaces
    // device workspace (one allocation, carved up)
    void *ws_base;
    int64_t ws_bytes;
    float2 *tw;            // [TW_N] twiddles
    float *tap_tab;        // [TAP_ROWS][32] constants of the taps of an image
    float *rir;            // [max_batch][max_sources][rir_taps]
    float2 *hspec;         // [max_batch][max_sources][n_part][CONV_BINS]
    float2 *xspec;         // [max_batch][max_sources][nblk_cap][CONV_BINS]; NULL unless route == ROUTE_STORED
    int nblk_cap;          // blocks of an utterance of max_samples
    float4 *park;          // [PARK_SLOTS][4096] products of noise sources waiting for the last one; NULL if unused
    int *park_flags;       // [PARK_SLOTS] 1 = slot held: that CTA sums in the time domain
    void *plans;           // [max_batch][PLAN_BYTES] what the fused convolution has to know of an utterance
    void *units;           // [2 unit_cap] its list of work
    int unit_cap;
    float *warped;         // [max_batch][ws_stride] speech after the waveform warp; NULL unless cfg.vtlp_win
    void *vtlp_tab;        // [max_batch][513] lower source bin (int), then [max_batch][513] fraction (float)
    float *ys;             // [max_batch][ws_stride]
    float *vv;             // [max_batch][ws_stride]
    double *energy;        // [max_batch][2]; this and the next two lie one behind the other, set to zero together
    unsigned long long *arrived;   // [max_batch] responses of callers: sources transformed and their lengths
    int *counters;         // [N_COUNTERS]
    int *leff;             // [max_batch][max_sources] taps of a response up to the last non-zero one
    int *leff_seen;        // pinned host copy of LEFF_ALL from an earlier call (long-response contexts)
    int stored_only;       // this call launches the stored-spectra kernels alone
    float *gain;           // [max_batch] noise gain g for the requested SNR
    aug::MelBin *melw;     // [max_batch][n_bins]
    int *melstart;         // [max_batch][n_mel + 2]
    int *status;           // [2]: utterance, reason
    // instrumentation
    int64_t launches;      // kernels launched so far
    int timing;            // record events between the stages of aug_pipeline
    cudaEvent_t *ev;       // [EV_RING][2 * AUG_N_STAGES]: start and stop of every stage
    int ev_n;              // calls recorded
    // staging for the host-buffer entry point (NULL unless cfg.host_staging)
    float *st_speech;      // [max_batch][ws_stride]
    float *st_bank;        // [max_bank_samples]
    AugUttParams *st_table;
    int *st_lengths;
    float *st_feats;       // [max_batch][t_cap][n_mel]
    int *st_counts;
    int64_t last_h2d, last_d2h;                // bytes the last aug_pipeline_host call copied
    cudaStream_t s_h2d, s_d2h;                 // copy streams of the host-buffer entry point
    cudaStream_t s_h2d2;                       // the row-gather kernel's stream, beside the copy engine's
    cudaEvent_t ev_in[aug::HOST_CHUNKS], ev_out[aug::HOST_CHUNKS], ev_start;
    cudaEvent_t ev_in2[aug::HOST_CHUNKS], ev_len;
    int64_t bank_resident;                     // samples of st_bank filled by aug_upload_noise_bank (0 = none)
};

#define AUG_CUDA_OK(expr)                         \
    do {                                          \
        cudaError_t e__ = (expr);                 \
        if (e__ != cudaSuccess) return AUG_ECUDA; \
    } while (0)

// Let kernel Kern use as much dynamic shared memory as the device allows (the
// opt-in limit less the kernel's static shared memory).  The attribute belongs to
// the device's copy of the kernel, not to a context, so it is set once per device
// and to the largest value any configuration can ask for.
template <auto Kern>
inline int smem_opt_in(int device) {
    static std::atomic<unsigned long long> done{0};
    const unsigned long long bit = 1ull << (device & 63);
    if (done.load(std::memory_order_acquire) & bit) return AUG_OK;
    int optin = 0;
    cudaFuncAttributes fa;
    AUG_CUDA_OK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
    AUG_CUDA_OK(cudaFuncGetAttributes(&fa, Kern));
    AUG_CUDA_OK(cudaFuncSetAttribute(Kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     optin - (int)fa.sharedSizeBytes));
    done.fetch_or(bit, std::memory_order_release);
    return AUG_OK;
}

// Kernels of aug_pipeline follow one another without the gap of a full launch: a chained kernel may
// start while the one before it on the stream is still running, as soon as all CTAs of that one
// have called chain_next() or ended (they call it towards their end: CTAs that arrive early and
// wait take room and slowed long kernels down, 1083 -> 1189 us on 128 x 8 s with 24000 taps); it calls
// chain_wait() before it touches anything an earlier kernel writes or reads.  As that one may be writing
// while this one lives, what it writes is not read through the non-coherent path (`const __restrict__`
// parameters, __ldg), which is for data that nobody writes meanwhile.  Every CTA of a chained kernel calls
// chain_wait() on every path, so that the end of a kernel implies the end of all before it.  (Both are no-ops in a
// kernel that was launched the ordinary way.)
#ifdef __CUDACC__
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename... P, typename... A>
inline int launch_chained(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...) == cudaSuccess ? AUG_OK : AUG_ECUDA;
}
#endif

// Whole part of n / by without a division: by a multiplication with 2^64 / by, rounded up.
struct Divisor {
    int by;
    unsigned long long m;
    explicit Divisor(int d) : by(d), m(~0ull / (unsigned)d + 1) {}      // (0 for 1)
#ifdef __CUDACC__
    __device__ __forceinline__ int of(int n) const { return by == 1 ? n : (int)__umul64hi((unsigned long long)n, m); }
#endif
};

// Where a kernel gets the noise gain from: worked out before (value), or from the two sums of the convolution.
struct GainSource {
    const float *value;             // [B], or NULL
    const double *energy;           // [B][2]
    const AugUttParams *table;
};
#ifdef __CUDACC__
// g = sqrt(sum y_s^2 / (sum v^2 10^(snr/10))), 0 without noise, with a silent side or with noise that is not
// finite, in fp64; `ratio` is 10^(snr/10).  -0 tells the feature kernel that v, though weighted by zero, is
// not silence (it may not be finite).
__device__ __forceinline__ bool snr_noisy(double es, double ev, int n_src) { return n_src > 1 && es > 0.0 && ev > 0.0; }
__device__ __forceinline__ float snr_gain(double es, double ev, double ratio, int n_src) {
    const float g = snr_noisy(es, ev, n_src) ? (float)sqrt(es / (ev * ratio)) : 0.f;
    return g == 0.f && ev != 0.0 ? -0.f : g;
}
__device__ __forceinline__ double snr_ratio(const AugUttParams &row) { return exp10((double)row.snr_db / 10.0); }
#endif

// What the convolution reads besides the responses; samples beyond max_len of a row are not used.
struct ConvInput {
    const float *speech;
    int64_t stride;
    const int *lengths;
    const float *bank;
    int64_t bank_len;
    int max_len;
    int room;              // CTAs of a full device left out for kernels that run beside the convolution
};

// Launchers (defined next to their kernels).  They enqueue on ctx->stream.
void rir_tap_table(int half_width, float *tab);
// `chained`: in aug_pipeline, behind launch_mel_tables; records where the responses end
int launch_rir(AugCtx *ctx, const AugUttParams *table, int B, float *rir, bool chained);
// `measured`: the responses come from launch_rir, which has recorded where they end (and launch_mel_tables has
// set the counters and sums of the convolution to zero); otherwise they are the caller's
int launch_rir_spectra(AugCtx *ctx, const float *rir, const ConvInput &in, const AugUttParams *table, int B,
                       bool measured);
// Convolution in two parts: `prepare` needs only the input audio (block spectra when
// the response has several partitions, else nothing), `finish` also needs the
// partition spectra of the impulse responses.
int launch_convolve_prepare(AugCtx *ctx, const ConvInput &in, const AugUttParams *table, int B, bool measured);
int launch_convolve_finish(AugCtx *ctx, const ConvInput &in, const AugUttParams *table, int B);
int launch_snr_gain(AugCtx *ctx, const AugUttParams *table, int B);
// `ready`: launch_snr_gain has been called
int launch_mix(AugCtx *ctx, const int *lengths, const AugUttParams *table, int B, int max_len, bool ready,
               float *wave_out, int64_t out_stride);
int launch_mel_tables(AugCtx *ctx, const AugUttParams *table, int B, bool reset);
int launch_vtlp_resynth(AugCtx *ctx, const float *speech, int64_t stride, const int *lengths,
                        const AugUttParams *table, int B, int max_len, float *out, int64_t out_stride);
int launch_stft_power(AugCtx *ctx, const float *wave, int64_t stride, const int *lengths, int B,
                      float *power, int T_max, int *counts);
int launch_logmel(AugCtx *ctx, const float *power, const int *counts, int B, int T_max,
                  float *feats);
bool features_write_wave(const AugCtx *ctx, int max_len, int T_max);
int launch_fused_features(AugCtx *ctx, const int *lengths, const AugUttParams *table, int B, float *feats, int T_max,
                          int *counts, int max_len, float *wave, int64_t wave_stride);
