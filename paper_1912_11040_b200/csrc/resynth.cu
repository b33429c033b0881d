// Waveform-domain VTLP: the warp of Eq. 1 applied to the speech itself, with
// resynthesis, before the simulator (Section 2.3; 50 ms window of Section 4).
//
// The paper prints only the frequency map.  The reading built here: frames of
// `win` samples every win/4, periodic Hann, the utterance zero-padded by
// win - win/4 samples in front; 1024-point DFT; the spectrum at bin k becomes the
// old spectrum at the frequency that Eq. 1 moves to bin k (the all-pass with the
// opposite coefficient), by linear interpolation between the two nearest bins;
// inverse DFT, first `win` samples, Hann again, overlap-add, division by the sum
// of the squared windows.
//
// A warp takes two frames through one pair of 512-point transforms and back (fft_pair.cuh):
// the (even, odd) sample pairs of a real frame are one complex signal of half the length.  The
// spectra are split off with the frequencies mirrored by shuffles, laid out in the warp's
// buffer (one 16-byte bin holds both frames), read back at the warped positions -- every lane
// both bins k and 512 - k, so that the inverse split needs the same shuffles only -- and
// transformed back; the windowed frames then replace the spectra in the buffer.  A CTA of
// eight warps does rounds of 16 consecutive frames.  Every output sample is covered by four
// frames: after a round the samples that have all four are written, what the round adds to
// the next three hops is carried over, so nothing is added across CTAs and only three frames
// per CTA are done twice.
//
// Bound by instruction issue.  The form before (64 threads per pair of frames as real and
// imaginary part of a 1024-point transform, scalar arithmetic, two exchanges and group
// barriers per transform, 16 frames for 13 hops) took 360 us for 64 utterances of 2-20 s, this
// one takes 261.  Its error is 1.8e-7 of the waveform (root mean square; the form before 2.3e-7); with
// the transforms' factors built from powers instead of a table it took 258 and had 3.1e-7.
#include <algorithm>

#include "common.cuh"
#include "fft_pair.cuh"

namespace {

using namespace fftpair;
constexpr int K = 1024;
constexpr int RS_THREADS = 256;
constexpr int NF = 2 * RS_THREADS / 32;        // frames per round
constexpr int SPEC = K / 2 + 1;                // bins
constexpr int WBUF = 2 * SPEC;                 // 8-byte words of a warp's buffer: spectra of both frames
static_assert(WBUF >= XBUF && 2 * WBUF >= 2 * K, "exchange and frames fit too");

// Shared memory, in floats.  (Passed to the kernel: offsets then cost no registers.)
struct ResynthLayout {
    int xin, win, pos, lanes, w512, carry, norm, total;
    explicit ResynthLayout(int w) {
        const int hop = w / 4;
        xin = 2 * WBUF * (RS_THREADS / 32);
        win = xin + (((NF - 1) * hop + w + 3) & ~3);
        pos = win + K;
        lanes = pos + 2 * SPEC + 2;
        w512 = (lanes + 6 * 32 + 3) & ~3;
        carry = w512 + 4 * 15 * 32;
        norm = carry + 3 * hop;              // (both on 16-byte boundaries where hops are multiples of 4)
        total = norm + hop;
    }
};

// Source position of every bin of an utterance: the frequency that Eq. 1 moves to bin k, in
// bins, as lower bin and fraction (fp64: a position error of 6e-5 bins, one fp32 ulp at bin 512,
// would already cost half of the waveform tolerance).
__global__ void __launch_bounds__(256)
vtlp_positions_kernel(const AugUttParams *__restrict__ table, int *__restrict__ k0_tab,
                      float *__restrict__ fr_tab) {
    const int utt = blockIdx.x;
    const double a = 1.0 - (double)table[utt].alpha;
    const double PI = 3.14159265358979323846;
    for (int k = threadIdx.x; k <= K / 2; k += 256) {
        const double om = 2.0 * PI * k / K;
        double pos = (om - 2.0 * atan(a * sin(om) / (1.0 + a * cos(om)))) * K / (2.0 * PI);
        if (k == 0) pos = 0.0;
        if (k == K / 2) pos = (double)(K / 2);
        int k0 = (int)floor(pos);
        k0 = min(max(k0, 0), K / 2 - 1);
        k0_tab[(int64_t)utt * SPEC + k] = k0;
        fr_tab[(int64_t)utt * SPEC + k] = (float)(pos - (double)k0);
    }
}

// Which hops a CTA owns: those of runs of several rounds or, in the utterances that come last, of single ones: the device is
// left half empty for a shorter time at the end (64 utterances of 2-20 s, warp and its tables 243 us, so 230).  Single
// rounds are a sixth more work, so no more utterances than two rounds for each place (4 of 100 s, window 400: 203 us in
// runs, 208 with one of them in single rounds).
struct HopMap {
    int long_utts;                 // utterances done in runs
    Divisor runs, singles;         // CTAs of an utterance in runs and in single rounds
};

// ROUNDS: rounds of a run; 1 where there are none (and the loop of rounds goes).
template <int ROUNDS>
__global__ void __launch_bounds__(RS_THREADS, 2)
vtlp_resynth_kernel(const float *__restrict__ speech, int64_t stride, const int *__restrict__ lengths,
                    const int *__restrict__ k0_tab, const float *__restrict__ fr_tab, int win,
                    const float2 *__restrict__ tw, float *__restrict__ out, int64_t out_stride, int n_cap,
                    const __grid_constant__ ResynthLayout lay, const HopMap map) {
    extern __shared__ __align__(16) float sm[];
    const int hop = win >> 2, front = win - hop;
    float *xin = sm + lay.xin;                       // [(NF-1) hop + win] padded input stretch of a round
    float *wn = sm + lay.win;                        // [K] Hann, zero beyond the window
    float2 *pos = reinterpret_cast<float2 *>(sm + lay.pos);      // [SPEC] lower source bin (int), fraction
    float *carry = sm + lay.carry;                   // [3 hop] what earlier frames add to the next hops

    int run = blockIdx.x, utt = map.runs.of(run), rounds = ROUNDS;
    if (utt < map.long_utts) {
        run -= utt * map.runs.by;
    } else {
        run -= map.long_utts * map.runs.by;
        utt = map.singles.of(run);
        run -= utt * map.singles.by;
        utt += map.long_utts;
        rounds = 1;
    }
    const int HB = rounds * NF - 3;                  // hops of output per CTA
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = min(max(lengths[utt], 0), n_cap);
    if (N == 0) return;
    const int T = (N + front + hop - 1) / hop;       // frames = hops that cover the padded utterance
    const int t0 = run * HB;                         // first hop this CTA owns
    if (t0 >= T) return;
    const float *x = speech + (int64_t)utt * stride;
    float *y = out + (int64_t)utt * out_stride;

    for (int k = tid; k < SPEC; k += RS_THREADS)
        pos[k] = make_float2(__int_as_float(k0_tab[(int64_t)utt * SPEC + k]), fr_tab[(int64_t)utt * SPEC + k]);
    for (int n = tid; n < K; n += RS_THREADS)
        wn[n] = n < win ? 0.5f - 0.5f * cospif(2.f * (float)n / (float)win) : 0.f;
    for (int i = tid; i < 3 * hop; i += RS_THREADS) carry[i] = 0.f;

    __syncthreads();
    // squared windows of the four frames over offset r of a hop; frames missing at the ends are left out below
    float *norm_s = sm + lay.norm;
    for (int i = tid; i < hop; i += RS_THREADS) {
        float norm = 0.f;
#pragma unroll
        for (int d = 0; d < 4; ++d) norm = fmaf(wn[i + d * hop], wn[i + d * hop], norm);
        norm_s[i] = norm;
    }

    u64 *buf = reinterpret_cast<u64 *>(sm) + warp * WBUF;
    const int mirror = (32 - lane) & 31;
    // lane constants of the transforms and the split; read again where they are used, as what follows
    // from them would otherwise be kept (and spilled) over the whole kernel
    float4 *lanes4 = reinterpret_cast<float4 *>(sm + lay.lanes);
    float2 *lanes2 = reinterpret_cast<float2 *>(lanes4 + 32);
    if (tid < 32) {
        const float2 w1 = __ldg(&tw[256 + tid]), wh = tid < 16 ? make_float2(1.f, 0.f) : __ldg(&tw[tid]);
        lanes4[tid] = make_float4(w1.x, w1.y, wh.x, wh.y);
        lanes2[tid] = __ldg(&tw[512 + tid]);         // exp(-2 pi i l / 1024)
    }
    // exp(-2 pi i l r / 512) at [r - 1][l], doubled
    float4 *w512 = reinterpret_cast<float4 *>(sm + lay.w512);
    for (int i = tid; i < 15 * 32; i += RS_THREADS) {
        const int k = ((i >> 5) + 1) * (i & 31);
        float2 w = __ldg(&tw[256 + (k & 255)]);
        if (k & 256) w = make_float2(-w.x, -w.y);
        w512[i] = make_float4(w.x, w.x, w.y, w.y);
    }

#pragma unroll 1
    for (int round = 0; round < rounds; ++round) {
        const int ft = t0 - 3 + round * NF;          // first frame of the round
        if (ft >= T) break;
        // input stretch of frames ft .. ft + NF - 1
        {
            const int at = ft * hop - front, n = (NF - 1) * hop + win;
            if (at >= 0 && at + n <= N) {
#pragma unroll 8
                for (int i = tid; i < n; i += RS_THREADS) xin[i] = __ldg(x + at + i);
            } else {
                for (int i = tid; i < n; i += RS_THREADS)
                    xin[i] = (at + i >= 0 && at + i < N) ? x[at + i] : 0.f;
            }
        }
        __syncthreads();
        const int fa = 2 * warp;                     // frame slots fa, fa + 1
        if (ft + fa + 1 >= 0 && ft + fa < T) {
            // (frames outside [0, T) are transformed with their neighbour but not added below)
            const float *c0 = xin + fa * hop, *c1 = c0 + hop;
            C2 v[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                v[r] = {0, 0};
                if (64 * r < win) {
                    // samples beyond the window are replaced by its last; their weight is zero
                    const int n = 2 * (lane + 32 * r);
                    const float2 w = *reinterpret_cast<const float2 *>(wn + n);
                    float2 p, q;
                    if ((hop & 1) == 0) {              // frames start on even samples
                        const int m = min(n, win - 2);
                        p = *reinterpret_cast<const float2 *>(c0 + m);
                        q = *reinterpret_cast<const float2 *>(c1 + m);
                    } else {
                        const int m = min(n, win - 1), o = min(n + 1, win - 1);
                        p = make_float2(c0[m], c0[o]);
                        q = make_float2(c1[m], c1[o]);
                    }
                    v[r] = {pack(w.x * p.x, w.x * q.x), pack(w.y * p.y, w.y * q.y)};
                }
            }
            fft512<true>(v, buf, lanes4[lane], lane, w512 + lane);

            // spectra (twice their value) of both frames into the buffer
            C2 mid = v[8];                           // lane 0: frequency 256
            if (lane == 0) {                         // its mirror images are its own points 16 - r
#pragma unroll
                for (int r = 8; r < 15; ++r) v[r] = v[r + 1];
                v[15] = v[0];
            }
            __syncwarp();
            // exp(-i pi r / 16)
            const float cr[8] = {1.f, 0.98078528040323044913f, 0.92387953251128675613f, 0.83146961230254523708f,
                                 0.70710678118654752440f, 0.55557023301960222474f, 0.38268343236508977173f,
                                 0.19509032201612826785f};
            const float ci[8] = {0.f, -0.19509032201612826785f, -0.38268343236508977173f, -0.55557023301960222474f,
                                 -0.70710678118654752440f, -0.83146961230254523708f, -0.92387953251128675613f,
                                 -0.98078528040323044913f};
            u64 *xr = buf, *xi = buf + SPEC;
            const float2 wl = lanes2[lane];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int k = lane + 32 * r;
                const C2 z = v[r], q = {shfl(v[15 - r].re, mirror), shfl(v[15 - r].im, mirror)};
                const u64 wx = both(fmaf(wl.x, cr[r], -wl.y * ci[r])), wy = both(fmaf(wl.x, ci[r], wl.y * cr[r]));
                const u64 evr = add2(z.re, q.re), evi = sub2(z.im, q.im), odr = add2(z.im, q.im), nodi = sub2(z.re, q.re);
                const u64 wor = fma2(wy, nodi, mul2(wx, odr)), woi = sub2(mul2(wy, odr), mul2(wx, nodi));
                xr[k] = add2(evr, wor);
                xi[k] = add2(evi, woi);
                xr[512 - k] = sub2(evr, wor);
                xi[512 - k] = sub2(woi, evi);
            }
            if (lane == 0) {
                const u64 two = both(2.f);
                xr[256] = mul2(two, mid.re);
                xi[256] = mul2(both(-2.f), mid.im);
            }
            __syncwarp();

            // the warped spectra, and back to the half-size transforms (four times their value), real
            // and imaginary parts swapped for the inverse
            auto warped = [&](int k) {
                const float2 s = pos[k];
                const int k0 = __float_as_int(s.x);
                const u64 fr = both(s.y), om = both(1.f - s.y);
                return C2{fma2(fr, xr[k0 + 1], mul2(om, xr[k0])), fma2(fr, xi[k0 + 1], mul2(om, xi[k0]))};
            };
            const float2 wm = lanes2[lane];
            if (lane == 0) {
                const C2 m = warped(256);
                mid = {mul2(both(-2.f), m.im), mul2(both(2.f), m.re)};
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int k = lane + 32 * r;
                const C2 a = warped(k), b = warped(512 - k);
                const u64 wx = both(fmaf(wm.x, cr[r], -wm.y * ci[r])), wy = both(fmaf(wm.x, ci[r], wm.y * cr[r]));
                const u64 ar = add2(a.re, b.re), ai = sub2(a.im, b.im), br = sub2(a.re, b.re), bi = add2(a.im, b.im);
                const u64 nqr = sub2(mul2(wx, bi), mul2(wy, br)), qi = fma2(wy, bi, mul2(wx, br));
                v[r] = {add2(ai, qi), sub2(ar, nqr)};
                v[15 - r] = {sub2(qi, ai), add2(ar, nqr)};
            }
#pragma unroll
            for (int r = 8; r < 16; ++r) v[r] = {shfl(v[r].re, mirror), shfl(v[r].im, mirror)};
            if (lane == 0) {
#pragma unroll
                for (int r = 15; r > 8; --r) v[r] = v[r - 1];
                v[8] = mid;
            }
            __syncwarp();                            // the buffer is free
            fft512<true>(v, buf, lanes4[lane], lane, w512 + lane);

            // both frames, windowed again, one behind the other
            float *fo = reinterpret_cast<float *>(buf);
            const float scale = 1.f / 2048.f;        // 4 from the splits, 512 from the transforms
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int n = 2 * (lane + 32 * r);
                if (n < win) {
                    const float2 w = *reinterpret_cast<const float2 *>(wn + n);
                    const float2 e = unpack(v[r].im), o = unpack(v[r].re);
                    *reinterpret_cast<float2 *>(fo + n) = make_float2(scale * w.x * e.x, scale * w.y * o.x);
                    *reinterpret_cast<float2 *>(fo + win + n) = make_float2(scale * w.x * e.y, scale * w.y * o.y);
                }
            }
        }
        __syncthreads();
        // Sample i of the round lies in hop q = i / hop at offset r; of the frames that cover it
        // (slots q - 3 .. q, at n = r + (q - slot) hop) this round holds slots 0 .. NF - 1, earlier ones
        // are in `carry` (first three hops).  Hops 0 .. NF - 1 are complete now.  Three loops: nothing of
        // `carry` is replaced before it has been read.
        const bool inner = ft >= 3 && ft + NF + 3 <= T;      // every frame that counts here exists
        auto add_up = [&](int i, int q) {
            float sum = 0.f;
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                const int slot = q - d, t = ft + slot;
                if ((unsigned)slot < (unsigned)NF && (inner || (t >= 0 && t < T)))
                    sum += sm[2 * WBUF * (slot >> 1) + (slot & 1) * win + i - q * hop + d * hop];
            }
            return sum;
        };
        const int first = round == 0 ? 3 : 0;        // (the hops before belong to the CTA before)
        const int at0 = ft * hop - front;            // utterance sample of i = 0
        if (inner && (hop & 3) == 0 && at0 + first * hop >= 0 && at0 + NF * hop <= N &&
            (reinterpret_cast<uintptr_t>(y) & 15) == 0) {
            // away from the utterance's ends four samples at a time: groups of four never cross a hop
            auto sum4 = [&](int g, int q) {
                float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    const int slot = q - d;
                    if ((unsigned)slot < (unsigned)NF) {
                        const float4 z = *reinterpret_cast<const float4 *>(
                            sm + 2 * WBUF * (slot >> 1) + (slot & 1) * win + 4 * g - (q - d) * hop);
                        sum = make_float4(sum.x + z.x, sum.y + z.y, sum.z + z.z, sum.w + z.w);
                    }
                }
                return sum;
            };
            const int hop4 = hop >> 2;
            const float inv = 1.f / (float)hop4;
            for (int g = first * hop4 + tid; g < NF * hop4; g += RS_THREADS) {
                const int q = (int)(((float)g + 0.5f) * inv);
                float4 z = sum4(g, q);
                if (q < 3) {
                    const float4 c = *reinterpret_cast<const float4 *>(carry + 4 * g);
                    z = make_float4(z.x + c.x, z.y + c.y, z.z + c.z, z.w + c.w);
                }
                const float4 n = *reinterpret_cast<const float4 *>(norm_s + 4 * g - q * hop);
                *reinterpret_cast<float4 *>(y + at0 + 4 * g) = make_float4(z.x / n.x, z.y / n.y, z.z / n.z, z.w / n.w);
            }
            __syncthreads();
            for (int g = tid; g < 3 * hop4; g += RS_THREADS)
                *reinterpret_cast<float4 *>(carry + 4 * g) = sum4(NF * hop4 + g, NF + (int)(((float)g + 0.5f) * inv));
            __syncthreads();
            continue;
        }
        for (int i = first * hop + tid; i < NF * hop; i += RS_THREADS) {
            const int q = (int)(((float)i + 0.5f) * (1.f / (float)hop));      // exact: i + 1/2 is never a multiple of hop
            const int c = ft * hop + i, idx = c - front;
            if (idx < 0 || idx >= N) continue;
            float sum = add_up(i, q);
            if (q < 3) sum += carry[i];
            float norm = norm_s[i - q * hop];
            if (!inner) {
                norm = 0.f;
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    const int t = ft + q - d;
                    if (t >= 0 && t < T) norm = fmaf(wn[c - t * hop], wn[c - t * hop], norm);
                }
            }
            y[idx] = sum / norm;
        }
        __syncthreads();
        for (int i = tid; i < 3 * hop; i += RS_THREADS)
            carry[i] = add_up(NF * hop + i, NF + (int)(((float)i + 0.5f) * (1.f / (float)hop)));
        __syncthreads();
    }
}

}  // namespace

int launch_vtlp_resynth(AugCtx *ctx, const float *speech, int64_t stride, const int *lengths,
                        const AugUttParams *table, int B, int max_len, float *out, int64_t out_stride) {
    const int win = ctx->cfg.vtlp_win;
    if (win <= 0 || max_len <= 0) return AUG_OK;
    const int hop = win / 4, front = win - hop;
    const int T_cap = (max_len + front + hop - 1) / hop;
    const ResynthLayout lay(win);
    const size_t smem = sizeof(float) * (size_t)lay.total;
    int *k0_tab = reinterpret_cast<int *>(ctx->vtlp_tab);
    float *fr_tab = reinterpret_cast<float *>(k0_tab + (size_t)ctx->cfg.max_batch * SPEC);
    vtlp_positions_kernel<<<B, 256, 0, ctx->stream>>>(table, k0_tab, fr_tab);
    AUG_CUDA_OK(cudaGetLastError());
    ctx->launches++;
    // Runs of three rounds (45 hops for 48 frames), single rounds (13 for 16) where the batch is so
    // small that it would not fill the device otherwise.
    constexpr int RUN = 3;
    HopMap map = {0, Divisor((T_cap + RUN * NF - 4) / (RUN * NF - 3)), Divisor((T_cap + NF - 4) / (NF - 3))};
    const bool runs = (int64_t)map.runs.by * B >= 4 * (int64_t)ctx->sm_count;
    if (runs) map.long_utts = std::max(0, B - 4 * ctx->sm_count / map.singles.by);
    auto kern = runs ? vtlp_resynth_kernel<RUN> : vtlp_resynth_kernel<1>;
    if ((runs ? smem_opt_in<vtlp_resynth_kernel<RUN>>(ctx->device) : smem_opt_in<vtlp_resynth_kernel<1>>(ctx->device)) !=
        AUG_OK)
        return AUG_ECUDA;
    const dim3 grid(map.long_utts * map.runs.by + (B - map.long_utts) * map.singles.by);
    kern<<<grid, RS_THREADS, smem, ctx->stream>>>(speech, stride, lengths, k0_tab, fr_tab, win, ctx->tw, out, out_stride,
                                                  max_len, lay, map);
    AUG_CUDA_OK(cudaGetLastError());
    ctx->launches++;
    return AUG_OK;
}
