// Steps 3 and 4: framing, Hann window, power spectrum, VTLP-warped mel
// filterbank and compression -- separately (frames_kernel<K, 0>, logmel_kernel) and
// fused with the SNR mix (frames_kernel<K, 1>: y_s + g v -> features, the power
// spectrum never leaves shared memory).
//
// The filterbank is applied as a gather: band m sums the bins of edge interval m
// with their rising weights and those of interval m+1 with their falling
// weights; the intervals are contiguous bin ranges because the warp of Eq. 1 is
// monotone.  Every interval is walked once for both sums.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "fft_pair.cuh"

namespace {

constexpr int FEAT_THREADS = 256;

__host__ __device__ __forceinline__ int frame_count(int n, int win, int hop) {
    return n >= win ? 1 + (n - win) / hop : 0;
}

// ---------------------------------------------------------------- filterbank tables
// Edges of the bands in mel: the first one and their distance.
struct MelEdges {
    double first, step;
    MelEdges(double f_lo, double f_hi, int M) {
        first = 2595.0 * log10(1.0 + f_lo / 700.0);
        step = (2595.0 * log10(1.0 + f_hi / 700.0) - first) / (M + 1);
    }
};
// One CTA per utterance: per DFT bin the edge interval and weights at the warped
// frequency (fp64: a bin that barely enters a band must not lose its weight to
// rounding), then the first bin of every interval.
__global__ void __launch_bounds__(256)
mel_tables_kernel(const AugUttParams *__restrict__ table, int K, int M, double fs, double e0, double delta,
                  aug::MelBin *__restrict__ melw, int *__restrict__ melstart, int unwarped, int *counters, double *energy) {
    __shared__ int seg_s[513];
    chain_next();
    // first kernel of aug_pipeline: the convolution's sums and counters start from zero
    if (energy != nullptr) {
        if (blockIdx.x == 0 && threadIdx.x < aug::N_COUNTERS) counters[threadIdx.x] = 0;
        if (threadIdx.x == 0) energy[2 * blockIdx.x] = energy[2 * blockIdx.x + 1] = 0.0;
    }
    const int utt = blockIdx.x, nb = K / 2 + 1;
    // (unwarped: the warp was already applied to the waveform)
    const double a = unwarped ? 0.0 : 1.0 - (double)table[utt].alpha;
    const double PI = 3.14159265358979323846;
    for (int k = threadIdx.x; k < nb; k += blockDim.x) {
        double sin_om, cos_om;
        sincospi(2.0 * k / K, &sin_om, &cos_om);
        const double omw = 2.0 * PI * k / K + 2.0 * atan(a * sin_om / (1.0 - a * cos_om));   // Eq. 1
        const double fw = omw * fs / (2.0 * PI);
        const double mu = 2595.0 * log10(1.0 + fw / 700.0);
        const double u = (mu - e0) / delta;
        int seg;
        aug::MelBin w;
        if (!(u >= 0.0)) {
            seg = -1;
            w.up = w.down = 0.f;
        } else if (u >= (double)(M + 1)) {
            seg = M + 1;
            w.up = w.down = 0.f;
        } else {
            const double fl = floor(u);
            seg = (int)fl;
            w.up = (float)(u - fl);
            w.down = (float)(1.0 - (u - fl));
        }
        seg_s[k] = seg;
        melw[(int64_t)utt * nb + k] = w;
    }
    int *st = melstart + (int64_t)utt * (M + 2);
    for (int m = threadIdx.x; m < M + 2; m += blockDim.x) st[m] = nb;
    __syncthreads();
    for (int k = threadIdx.x; k < nb; k += blockDim.x) {
        const int prev = k ? seg_s[k - 1] : -1;
        const int cur = seg_s[k];
        for (int m = prev + 1; m <= cur && m < M + 2; ++m) st[m] = k;   // first bin with seg >= m
    }
}

// n floats of value `val` from dst on by the threads of a CTA, 128 bits at a time where they can be.
__device__ __forceinline__ void fill_floats(float *dst, int n, float val, int tid, int threads) {
    const int head = min(n, (int)((4 - ((reinterpret_cast<uintptr_t>(dst) >> 2) & 3)) & 3));
    if (tid < head) dst[tid] = val;
    const int n4 = (n - head) >> 2;
    for (int i = tid; i < n4; i += threads)
        reinterpret_cast<float4 *>(dst + head)[i] = make_float4(val, val, val, val);
    const int tail = head + 4 * n4 + tid;
    if (tail < n) dst[tail] = val;
}

__device__ __forceinline__ float compress(float e, float floor_v, int mode) {
    e = fmaxf(e, floor_v);
    const float l = logf(e);
    return mode == AUG_COMPRESS_LOG ? l : expf(l * (1.f / 15.f));
}

// ---------------------------------------------------------------- filterbank
// Bands are dealt out in RUNS runs of consecutive ones, cut so that all cost about the same: a band
// costs its bins and about four bins' worth of set-up.  By the first RUNS + 1 threads.
template <int RUNS>
__device__ __forceinline__ void cut_bands(int *cut, const int *mst, int M, int tid) {
    if (tid > RUNS) return;
    const int base = mst[0], total = mst[M + 1] - base + 4 * M, want = total * tid / RUNS;
    int lo = 0, hi = M;
    while (lo < hi) {
        const int m = (lo + hi) >> 1;
        if (mst[m] - base + 4 * m < want) lo = m + 1;
        else hi = m;
    }
    cut[tid] = tid == RUNS ? M : lo;
}
// Where the powers of two frames come from: words that hold both, or two rows of floats.
struct PairRow {
    const fftpair::u64 *p;
    __device__ __forceinline__ fftpair::u64 at(int i) const { return p[i]; }
    __device__ __forceinline__ void step(int n) { p += n; }
};
struct TwoRows {
    const float *p;
    int next;
    __device__ __forceinline__ fftpair::u64 at(int i) const { return fftpair::pack(p[i], p[next + i]); }
    __device__ __forceinline__ void step(int n) { p += n; }
};
// Energies of bands m0 .. m1 - 1 of two frames: w4[k] the doubled weights of bin k (rising, falling),
// `power` at bin 0, fs[m] and fs[m + next] the results.  The bins of edge interval j
// give the falling sum of band j - 1 and the rising sum of band j.
template <typename Power>
__device__ __forceinline__ void walk_bands(const ulonglong2 *w4, const int *mst, int m0, int m1, Power power,
                                           float *fs, int next) {
    using namespace fftpair;
    if (m0 >= m1) return;
    int k = mst[m0];
    w4 += k;
    power.step(k);
    fs += m0;
    u64 u = 0, d = 0;              // rising and falling sums
    auto walk = [&](int j) {
        int n = mst[j + 1] - k;
        k += n;
#pragma unroll 1
        for (; n >= 2; n -= 2, w4 += 2, power.step(2)) {
            const ulonglong2 wa = w4[0], wb = w4[1];
            const u64 pa = power.at(0), pb = power.at(1);
            u = fma2(wa.x, pa, u);
            d = fma2(wa.y, pa, d);
            u = fma2(wb.x, pb, u);
            d = fma2(wb.y, pb, d);
        }
        if (n > 0) {
            const ulonglong2 wa = *w4++;
            const u64 pa = power.at(0);
            power.step(1);
            u = fma2(wa.x, pa, u);
            d = fma2(wa.y, pa, d);
        }
    };
    walk(m0);
#pragma unroll 1
    for (int j = m0 + 1; j <= m1; ++j) {
        d = u;                     // rising sum of band j - 1, to which its falling one is added
        u = 0;
        walk(j);
        const float2 e = unpack(d);
        fs[0] = e.x;
        fs[next] = e.y;
        ++fs;
    }
}

// ---------------------------------------------------------------- frames -> spectra -> features
// A warp takes four frames (512-point transform) or two (1024) from their samples to their
// power spectra with one pair of 512-point transforms (fft_pair.cuh):
//   K = 512   transform A holds frames 0 and 1 as real and imaginary part, B frames 2 and 3
//   K = 1024  transform A holds the (even, odd) sample pairs of frame 0, B those of frame 1
// Afterwards lane l holds the frequencies l + 32 r; the mirrored ones come from lane
// (32 - l) mod 32 by shuffles, the spectra are separated and squared in registers, and the
// powers replace the exchange buffer of the warp.  A CTA of eight warps does a tile of FT
// frames at a time; the filterbank then runs with the frames of the tile over the lanes.
// Every group of FT lanes walks a run of consecutive bands, cut so that all runs cover about
// as many bins: the bins of edge interval j give the falling sum of band j - 1 and the rising
// sum of band j, so each band is finished in registers.  The samples of the next tile are
// already on their way from global memory meanwhile.
//
// Bound by the issue of instructions.  The kernel this replaced (a pair of frames per warp,
// scalar arithmetic, three radix-8 passes with two exchanges through shared memory, band sums
// in shared memory) issued 829 warp instructions a frame: 295 us on 256 utterances of 2-20 s
// (K = 512, 40 bands) where this one takes 249, and 874 against 653 on 64 of 60 s (K = 1024, 128
// bands); the bytes take 61 and 105.  Tiles of a run, on the former batch and on 4096 of 1-6 s: two
// 264 and 1302 us, four 249 and 1179, six 249 and 1190.
constexpr int WARPS = FEAT_THREADS / 32;
constexpr int TAIL_ROUNDS = 2;         // tiles a CTA's place on the device that are not done in runs
constexpr int TAIL_SAMPLES = 8192;     // samples of a large tile, see launch_frames

template <int K>
struct Plan;
template <>
struct Plan<512> {
    static constexpr int QF = 4, TILES = 4;           // frames per warp; tiles of a run
};
template <>
struct Plan<1024> {
    static constexpr int QF = 2, TILES = 8;
};
template <int K>
__host__ __device__ constexpr int tile_frames() { return WARPS * Plan<K>::QF; }

// Floats of a warp's buffer: 2 XBUF for the exchange, or its power rows.  A multiple of 32
// plus 4, and odd rows, so that the frames of a tile start at different banks.
constexpr int SPAN = 1092;
static_assert(SPAN >= 2 * fftpair::XBUF && SPAN >= 4 * 257 && SPAN >= 2 * 513 && SPAN % 32 == 4, "");
// Powers lie in pairs, as the arithmetic leaves them: one 64-bit word holds a bin of frames
// 4 w and 4 w + 2 (row 0 of warp w) or 4 w + 1 and 4 w + 3 (row 1); K = 1024: 2 w and 2 w + 1.

// Shared memory, in floats.  MODE 0: wave -> power.  MODE 1: y_s + g v -> features.
//   AHEAD    the next tile is copied in while the current one is worked on
//   DIRECT   there is one tile buffer, filled when it is needed
//   PACKED   so too, and without the gaps that hops longer than the window leave between the frames
enum Staging { AHEAD, DIRECT, PACKED };
struct Layout {
    int chunk_cap;      // samples of a tile, in whole groups of 4
    int step;           // between the frames of a tile in its buffer
    int fs_ld;          // row stride of a tile's band energies
    int ahead, packed;
    int chunk, raw, win, lanes, mw, mst, cut, total;
};
// Frames lie at the same offset from a 16-byte boundary as in their row, and so far apart that the
// groups at the ends of two neighbours do not meet.
inline int packed_step(int win_len, int hop) { return win_len + 6 + ((hop - win_len - 6) & 3); }
template <int K, int MODE>
Layout make_layout(int win_len, int hop, int M, Staging staging) {
    constexpr int FT = tile_frames<K>();
    const bool ahead = staging == AHEAD;
    Layout l;
    l.ahead = ahead;
    l.packed = staging == PACKED;
    l.step = l.packed ? packed_step(win_len, hop) : hop;
    l.fs_ld = M | 1;
    // (where tiles begin anywhere, up to three samples before the first one come along)
    l.chunk_cap = ((FT - 1) * l.step + win_len + ((hop & 3) ? 3 : 0) + 3) & ~3;
    int o = WARPS * SPAN;
    auto take = [&](int n) { const int r = o; o = (o + n + 3) & ~3; return r; };
    // samples of the tile; later (MODE 1) its band energies
    l.chunk = take(MODE == 1 && FT * l.fs_ld > l.chunk_cap ? FT * l.fs_ld : l.chunk_cap);
    l.raw = take(!ahead ? 0 : (MODE == 1 ? 2 : 1) * l.chunk_cap);   // MODE 0: the next tile; MODE 1: its y_s and v
    l.win = take(K);
    l.lanes = take(4 * 32);
    l.mw = take(MODE == 1 ? 4 * (K / 2 + 1) : 0);
    l.mst = take(MODE == 1 ? M + 2 : 0);
    l.cut = take(MODE == 1 ? 64 : 0);            // (the last one: the gain)
    l.total = o;
    return l;
}

// 16 bytes global -> shared without passing through registers; beyond `bytes`: zeros.
__device__ __forceinline__ void copy16_async(float *dst_smem, const float *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst_smem)),
                 "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The samples of a warp's frames, windowed, as the points l + 32 r of a transform pair.
template <int K>
__device__ __forceinline__ void windowed_points(fftpair::C2 *v, const float *c0, const float *win_s, int win,
                                                int step, int l) {
    using namespace fftpair;
    const float *c1 = c0 + step, *c2 = c1 + step, *c3 = c2 + step;   // (K = 512: four frames)
    auto point = [&](int i, int j, float2 w) {                       // samples i (and i + 1 = j) of every frame
        if (K == 512) {
            const u64 ww = both(w.x);
            return C2{mul2(ww, pack(c0[i], c2[i])), mul2(ww, pack(c1[i], c3[i]))};
        }
        return C2{pack(w.x * c0[i], w.x * c1[i]), pack(w.y * c0[j], w.y * c1[j])};
    };
    constexpr int SP = K / 512;                                      // samples per point
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int n = SP * (l + 32 * r);
        if (SP * 32 * (r + 1) <= win) {
            v[r] = point(n, n + 1, K == 512 ? make_float2(win_s[n], 0.f) : *reinterpret_cast<const float2 *>(win_s + n));
        } else if (SP * 32 * r < win) {
            // a sample beyond the window is replaced by the window's last; its weight is zero
            v[r] = point(min(n, win - 1), min(n + 1, win - 1),
                         K == 512 ? make_float2(win_s[n], 0.f) : *reinterpret_cast<const float2 *>(win_s + n));
        } else {
            v[r] = {0, 0};
        }
    }
}

// Power spectra of a warp's frames from the frequencies l + 32 r in v (of samples that carry
// the window at half its height) into the warp's rows at p.
template <int K>
__device__ __forceinline__ void power_rows(fftpair::C2 *v, fftpair::u64 *p, const float2 *__restrict__ tw, int l) {
    using namespace fftpair;
    constexpr int NBP = K / 2 + 1;
    const C2 mid = v[8];                             // lane 0: frequency 256
    const int mirror = (32 - l) & 31;
    if (l == 0) {                                    // its mirror images are its own points 16 - r
#pragma unroll
        for (int r = 8; r < 15; ++r) v[r] = v[r + 1];
        v[15] = v[0];
    }
    __syncwarp();
    const float2 wl = K == 1024 ? __ldg(&tw[512 + l]) : make_float2(0.f, 0.f);       // exp(-2 pi i l / 1024)
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const C2 z = v[r], q = {shfl(v[15 - r].re, mirror), shfl(v[15 - r].im, mirror)};
        const u64 ar = add2(z.re, q.re), ai = sub2(z.im, q.im), br = add2(z.im, q.im), bi = sub2(z.re, q.re);
        const int k = l + 32 * r;
        if (K == 512) {
            p[k] = fma2(ar, ar, mul2(ai, ai));
            p[NBP + k] = fma2(br, br, mul2(bi, bi));
        } else {
            // even part (ar, ai), odd part (br, -bi), joined with W = exp(-2 pi i k / 1024)
            // exp(-i pi r / 16)
            const float cr[8] = {1.f, 0.98078528040323044913f, 0.92387953251128675613f, 0.83146961230254523708f,
                                 0.70710678118654752440f, 0.55557023301960222474f, 0.38268343236508977173f,
                                 0.19509032201612826785f};
            const float ci[8] = {0.f, -0.19509032201612826785f, -0.38268343236508977173f, -0.55557023301960222474f,
                                 -0.70710678118654752440f, -0.83146961230254523708f, -0.92387953251128675613f,
                                 -0.98078528040323044913f};
            const u64 wx = both(fmaf(wl.x, cr[r], -wl.y * ci[r])), wy = both(fmaf(wl.x, ci[r], wl.y * cr[r]));
            const u64 tr = fma2(wy, bi, mul2(wx, br)), ti = sub2(mul2(wy, br), mul2(wx, bi));
            const u64 xr = add2(ar, tr), xi = add2(ai, ti), yr = sub2(ar, tr), yi = sub2(ai, ti);
            p[k] = fma2(xr, xr, mul2(xi, xi));
            p[512 - k] = fma2(yr, yr, mul2(yi, yi));
        }
    }
    if (l == 0) {
        const u64 four = both(4.f), re2 = mul2(four, mul2(mid.re, mid.re)), im2 = mul2(mid.im, mid.im);
        if (K == 512) {
            p[256] = re2;
            p[NBP + 256] = mul2(four, im2);
        } else {
            p[256] = fma2(four, im2, re2);
        }
    }
}

// Which frames a CTA works on.  Runs of several tiles share their set-up, but the device is left half empty behind the
// last round of them; the utterances that come last are done tile by tile.  The last utterances go first: what the
// convolution has written last is still in L2.  256 utterances of 2-20 s 258 -> 252 us, 96 116 -> 112, 64 of 60 s (K = 1024)
// 666 -> 649; with twice as many single tiles 686.2 against 689.3 and 1376 against 1373 (whole calls), with four times as
// many both slower.
struct RunMap {
    int utts, long_utts;           // of which the first ones (in the order of work) are done in runs
    Divisor runs, tiles;           // per utterance: runs, tiles
};

// TILES: tiles of a run; 1 where there are none, so that no loop and no arithmetic of runs is left.
template <int K, int MODE, int TILES>
__global__ void __launch_bounds__(FEAT_THREADS, 2)
frames_kernel(const float *in_a, const float *in_b, int64_t in_stride, const GainSource gain,
              const int *__restrict__ lengths, int win, int hop, int M, int T_max, const aug::MelBin *__restrict__ melw,
              const int *__restrict__ melstart, const float2 *__restrict__ tw, float floor_v, float pad_v, int comp,
              float *__restrict__ out, int *__restrict__ counts, int n_cap, float *__restrict__ wave, int64_t wave_stride,
              const __grid_constant__ Layout lay, const RunMap map) {
    constexpr int QF = Plan<K>::QF, FT = tile_frames<K>(), NBP = K / 2 + 1;
    extern __shared__ __align__(16) float sm[];
    float *chunk = sm + lay.chunk, *win_s = sm + lay.win;
    float4 *mw = reinterpret_cast<float4 *>(sm + lay.mw);                    // (up, up, down, down)
    int *mst = reinterpret_cast<int *>(sm + lay.mst), *cut = reinterpret_cast<int *>(sm + lay.cut);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // (single tiles throughout: two grid dimensions.  With the same arithmetic for all, divisions in it, the power
    // spectra of one utterance of 3 s took 8.2 us instead of 7.2)
    int run = blockIdx.x, nth = blockIdx.y, run_tiles = TILES;
    if (TILES > 1) {
        nth = map.runs.of(run);
        if (nth < map.long_utts) {
            run -= nth * map.runs.by;
        } else {
            run -= map.long_utts * map.runs.by;
            nth = map.tiles.of(run);
            run -= nth * map.tiles.by;
            nth += map.long_utts;
            run_tiles = 1;
        }
    }
    const int utt = map.utts - 1 - nth, run0 = run * (FT * run_tiles);
    for (int n = tid; n < K; n += FEAT_THREADS)
        win_s[n] = n < win ? 0.25f - 0.25f * cospif(2.f * (float)n / (float)win) : 0.f;
    if (tid < 32) {
        const float2 w1 = __ldg(&tw[256 + tid]), wh = tid < 16 ? make_float2(1.f, 0.f) : __ldg(&tw[tid]);
        reinterpret_cast<float4 *>(sm + lay.lanes)[tid] = make_float4(w1.x, w1.y, wh.x, wh.y);
    }
    const int N = min(max(lengths[utt], 0), n_cap);
    const int T = min(frame_count(N, win, hop), T_max);
    if (run == 0 && tid == 0) counts[utt] = T;
    const int rows = min(FT * run_tiles, T_max - run0);
    const int nfr = max(0, min(FT * run_tiles, T - run0));
    const int out_w = MODE == 0 ? NBP : M;
    float *orun = out + ((int64_t)utt * T_max + run0) * out_w;
    if (rows > nfr)
        fill_floats(orun + (int64_t)nfr * out_w, (rows - nfr) * out_w, MODE == 0 ? 0.f : pad_v, tid, FEAT_THREADS);
    // The gain is one thread's work, done while the first tile's samples travel.
    const bool gains = MODE == 1 && tid == FEAT_THREADS - 1;
    const double ratio = gains ? snr_ratio(gain.table[utt]) : 1.0;
    const int n_src = MODE == 1 ? gain.table[utt].n_src : 0;
    chain_wait();
    double es = 0.0, ev = 0.0;
    if (MODE == 1) {
        es = gain.energy[2 * utt];
        ev = gain.energy[2 * utt + 1];
    }
    float g = 0.f, *gain_s = sm + lay.cut + 63;
    bool noisy = MODE == 1 && snr_noisy(es, ev, n_src);      // v is copied
    // The mixed waveform, where it is wanted: a tile writes the hops that its frames start, the CTA with
    // the last frame (the first one if there is none) what lies behind them.
    float *wrow = MODE == 1 && wave != nullptr ? wave + (int64_t)utt * wave_stride : nullptr;
    if (MODE == 1 && wrow != nullptr && run0 <= max(T - 1, 0) && run0 + FT * run_tiles > max(T - 1, 0)) {
        const float gw = fabsf(snr_gain(es, ev, snr_ratio(gain.table[utt]), n_src));
        const float *wa = in_a + (int64_t)utt * in_stride, *wb = in_b + (int64_t)utt * in_stride;
        for (int i = T * hop + tid; i < N; i += FEAT_THREADS) wrow[i] = fmaf(gw, wb[i], wa[i]);
    }
    if (nfr == 0) return;

    const float *ra = in_a + (int64_t)utt * in_stride;
    const float *rb = MODE == 1 ? in_b + (int64_t)utt * in_stride : nullptr;
    const int n_tiles = min(run_tiles, (nfr + FT - 1) / FT);

    // Samples of a tile travel global -> shared asynchronously, one tile ahead, in the 16-byte groups of
    // the row: the tile's first sample may be any of its first group (with hops that are no
    // multiple of 4, one sample after another and one tile at a time, 128 utterances of 10 s took 506 us
    // at K = 1024 and a hop of 441, and 471 at K = 512 and 125; so 322 and 315).  MODE 1: a thread
    // copies the groups 4 (tid + 256 u) of y_s and v into the raw buffers, and one tile
    // later mixes the same groups into `chunk`, so the raw slots are private to the thread and need
    // no barrier.  MODE 0 copies into the two tile buffers in turn.  Beyond the frames there are: zeros.
    auto stage_issue = [&](int tile) {
        const int t0 = run0 + tile * FT, off = (t0 * hop) & 3, s0 = t0 * hop - off;
        const int ns = (min(FT, T - t0) - 1) * hop + win + off;
        float *a = MODE == 1 ? sm + lay.raw : sm + ((tile & 1) ? lay.raw : lay.chunk), *b = a + lay.chunk_cap;
        if (t0 + FT <= T) {
            // a full tile: whole groups (rows are allocated up to a multiple of 4 floats), what the last
            // one holds beyond the tile is not used
            const float *pa = ra + s0, *pb = rb + s0;
#pragma unroll 2
            for (int i = 4 * tid; i < ns; i += 4 * FEAT_THREADS) {
                copy16_async(a + i, pa + i, 16);
                if (noisy) copy16_async(b + i, pb + i, 16);
            }
            return;
        }
        for (int i = 4 * tid; i < lay.chunk_cap; i += 4 * FEAT_THREADS) {
            const int bytes = 4 * min(max(ns - i, 0), 4), src = bytes ? s0 + i : 0;
            copy16_async(a + i, ra + src, bytes);
            if (noisy) copy16_async(b + i, rb + src, bytes);
        }
    };
    auto stage_mix = [&]() {
        const float *a = sm + lay.raw, *b = a + lay.chunk_cap;
        for (int i = 4 * tid; i < lay.chunk_cap; i += 4 * FEAT_THREADS) {
            float4 x = *reinterpret_cast<const float4 *>(a + i);
            if (noisy) {
                const float4 y = *reinterpret_cast<const float4 *>(b + i);
                x = make_float4(fmaf(g, y.x, x.x), fmaf(g, y.y, x.y), fmaf(g, y.z, x.z), fmaf(g, y.w, x.w));
            }
            *reinterpret_cast<float4 *>(chunk + i) = x;
        }
    };
    // Where there is one tile buffer: n samples from sample s0 on to chunk[d0], by every `step`-th thread
    // from `first` on.  Whole groups, four loads (of each array) in flight, where rows hold such.
    const bool groups = (in_stride & 3) == 0;
    auto stage_stretch = [&](int s0, int d0, int n, int first, int step) {
        if (groups) {
            const int lead = s0 & 3, n4 = (lead + n + 3) >> 2;         // (d0 has the same lead)
            const float4 *pa = reinterpret_cast<const float4 *>(ra + s0 - lead);
            const float4 *pb = reinterpret_cast<const float4 *>(rb + s0 - lead);
            float4 *d = reinterpret_cast<float4 *>(chunk + d0 - lead);
            for (int i = first; i < n4; i += 4 * step) {
                float4 x[4], y[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    x[u] = y[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (i + u * step < n4) {
                        x[u] = pa[i + u * step];
                        if (noisy) y[u] = pb[i + u * step];
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (i + u * step < n4)
                        d[i + u * step] = !noisy ? x[u] : make_float4(fmaf(g, y[u].x, x[u].x), fmaf(g, y[u].y, x[u].y),
                                                                      fmaf(g, y[u].z, x[u].z), fmaf(g, y[u].w, x[u].w));
            }
        } else {
#pragma unroll 4
            for (int i = first; i < n; i += step) chunk[d0 + i] = noisy ? fmaf(g, rb[s0 + i], ra[s0 + i]) : ra[s0 + i];
        }
    };
    auto stage_direct = [&](int tile) {
        const int t0 = run0 + tile * FT, s0 = t0 * hop, off = groups ? s0 & 3 : 0, nf = min(FT, T - t0);
        if (lay.packed) {
            for (int f = warp; f < nf; f += WARPS) stage_stretch(s0 + f * hop, off + f * lay.step, win, lane, 32);
        } else {
            stage_stretch(s0, off, (nf - 1) * hop + win, tid, FEAT_THREADS);
        }
        // frames that there are not are transformed beside others: zeros
        if (nf < FT) {
            const int end = off + (nf - 1) * lay.step + win;
            __syncthreads();                  // (the last group may reach beyond the last frame)
            for (int i = end + tid; i < lay.chunk_cap; i += FEAT_THREADS) chunk[i] = 0.f;
        }
    };
    if (lay.ahead) stage_issue(0);

    constexpr int RUNS = 2 * FEAT_THREADS / FT;       // runs of bands, one per FT / 2 lanes
    if (MODE == 1) {
        if (gains) *gain_s = snr_gain(es, ev, ratio, n_src);
        for (int k = tid; k < NBP; k += FEAT_THREADS) {
            const aug::MelBin w = melw[(int64_t)utt * NBP + k];
            mw[k] = make_float4(w.up, w.up, w.down, w.down);
        }
        for (int m = tid; m < M + 2; m += FEAT_THREADS) mst[m] = melstart[(int64_t)utt * (M + 2) + m];
        __syncthreads();
        cut_bands<RUNS>(cut, mst, M, tid);
        g = *gain_s;
        noisy = noisy && g != 0.f;            // (0 beside an infinite sum: v may hold an infinity, is not read)
    }
    fftpair::u64 *xb = reinterpret_cast<fftpair::u64 *>(sm + warp * SPAN);

    for (int tile = 0; tile < n_tiles; ++tile) {
        const int t0 = run0 + tile * FT;
        const int nf = min(FT, T - t0);
        const int off = groups ? (t0 * hop) & 3 : 0;          // of the tile's first sample in its buffer
        if (lay.ahead) {
            copies_done();
            if (MODE == 1) {
                stage_mix();
                if (tile + 1 < n_tiles) stage_issue(tile + 1);
            }
        } else {
            stage_direct(tile);
        }
        __syncthreads();                      // samples (and, first time, the tables) in place
        if (MODE == 1 && wrow != nullptr) {
            float *o = wrow + t0 * hop;
            const int n = nf * hop;
            const bool vec = ((hop | (int)wave_stride) & 3) == 0 && (reinterpret_cast<uintptr_t>(wave) & 15) == 0;
            const float *pa = ra + t0 * hop, *pb = rb + t0 * hop;
            if (__float_as_int(g) < 0) {
                // -0, see snr_gain: noise that is not finite shows in the waveform, though the features
                // (of y_s alone) never read it.  (Done for every utterance without noise it cost 4 % of 96
                // utterances of 2-20 s.)
                if (vec) {
#pragma unroll 2
                    for (int i = 4 * tid; i < n; i += 4 * FEAT_THREADS) {
                        const float4 x = *reinterpret_cast<const float4 *>(pa + i), y = *reinterpret_cast<const float4 *>(pb + i);
                        *reinterpret_cast<float4 *>(o + i) =
                            make_float4(fmaf(0.f, y.x, x.x), fmaf(0.f, y.y, x.y), fmaf(0.f, y.z, x.z), fmaf(0.f, y.w, x.w));
                    }
                } else {
                    for (int i = tid; i < n; i += FEAT_THREADS) o[i] = fmaf(0.f, pb[i], pa[i]);
                }
            } else if (vec) {
                for (int i = 4 * tid; i < n; i += 4 * FEAT_THREADS)
                    *reinterpret_cast<float4 *>(o + i) = *reinterpret_cast<const float4 *>(chunk + i);
            } else {
                for (int i = tid; i < n; i += FEAT_THREADS) o[i] = chunk[off + i];
            }
        }
        if (MODE == 0 && lay.ahead && tile + 1 < n_tiles) stage_issue(tile + 1);

        const int f0 = QF * warp;
        if (f0 < nf) {
            fftpair::C2 v[16];
            const float *c0 = (MODE == 0 && lay.ahead && (tile & 1) ? sm + lay.raw : chunk) + off + f0 * lay.step;
            windowed_points<K>(v, c0, win_s, win, lay.step, lane);
            fftpair::fft512<false>(v, xb, reinterpret_cast<const float4 *>(sm + lay.lanes)[lane], lane);
            power_rows<K>(v, xb, tw, lane);
            if (MODE == 0) {
                __syncwarp();
                float *o = orun + (int64_t)(tile * FT + f0) * NBP + lane;
#pragma unroll
                for (int q = 0; q < QF / 2; ++q) {
                    const bool first = f0 + q < nf, second = f0 + q + QF / 2 < nf;
#pragma unroll
                    for (int i = 0; i < (NBP + 31) / 32; ++i) {
                        if (32 * i + lane < NBP) {
                            const float2 z = fftpair::unpack(xb[q * NBP + 32 * i + lane]);
                            if (first) o[q * NBP + 32 * i] = z.x;
                            if (second) o[(q + QF / 2) * NBP + 32 * i] = z.y;
                        }
                    }
                }
                __syncwarp();
            }
        }
        if (MODE == 0) {
            if (!lay.ahead) __syncthreads();      // the one tile buffer is rewritten
            continue;
        }
        __syncthreads();                      // power spectra of the tile in place

        {
            using namespace fftpair;
            constexpr int PT = FT / 2;               // frame pairs of the tile
            const int pr = tid & (PT - 1), run = tid / PT, w = pr / (QF / 2), q = pr % (QF / 2);
            const int f = QF * w + q;                // and f + QF / 2
            if (f < nf) {
                walk_bands(reinterpret_cast<const ulonglong2 *>(mw), mst, cut[run], cut[run + 1],
                           PairRow{reinterpret_cast<const u64 *>(sm + w * SPAN) + q * NBP}, chunk + f * lay.fs_ld,
                           (QF / 2) * lay.fs_ld);
            }
        }
        __syncthreads();                      // band energies in place
        float *orow = orun + (int64_t)tile * FT * M;
        auto value = [&](float e) {
            e = fmaxf(e, floor_v);
            if (K == 1024) {
                const float l = logf(e);
                return comp == AUG_COMPRESS_LOG ? l : expf(l * (1.f / 15.f));
            }
            const float l = __logf(e);
            return comp == AUG_COMPRESS_LOG ? l : __expf(l * (1.f / 15.f));
        };
        if ((M & 3) == 0) {
            const int m4 = M >> 2, step_f = FEAT_THREADS / m4, step_m = FEAT_THREADS - step_f * m4;
            int f = tid / m4, m = tid - f * m4;
            for (int i = tid; i < nf * m4; i += FEAT_THREADS) {
                const float *e = chunk + f * lay.fs_ld + 4 * m;
                reinterpret_cast<float4 *>(orow)[i] = make_float4(value(e[0]), value(e[1]), value(e[2]), value(e[3]));
                f += step_f;
                m += step_m;
                if (m >= m4) {
                    m -= m4;
                    ++f;
                }
            }
        } else {
            for (int i = tid; i < nf * M; i += FEAT_THREADS) {
                const int f = i / M;
                orow[i] = value(chunk[i + f * (lay.fs_ld - M)]);
            }
        }
        __syncthreads();                      // the features' place is the next tile's
    }
}

// ---------------------------------------------------------------- step 4 alone
// A CTA copies a tile of 32 frames, which are contiguous, into shared memory (16-byte asynchronous
// copies; the tile starts at the same offset from a 16-byte boundary as in global memory) and walks
// the filterbank as the fused kernels do, half a warp per run of bands, two frames a lane.
// Bound by issue: 80 bands, 205 k frames 86 us where the bytes take 51; with one frame a lane and
// the interval sums in shared memory 101, gathered from global memory one thread per band and
// frame 203.
constexpr int LM_FT = 32, LM_RUNS = 16;
__host__ __device__ constexpr int logmel_fs(int NBP) { return ((LM_FT * NBP + 4) + 3) & ~3; }
__host__ __device__ constexpr int logmel_mw(int NBP, int M) { return (logmel_fs(NBP) + LM_FT * (M | 1) + 3) & ~3; }
__host__ __device__ constexpr size_t logmel_smem(int NBP, int M) {
    return sizeof(float) * (size_t)(logmel_mw(NBP, M) + 4 * NBP + M + 2 + LM_RUNS + 1);
}
__global__ void __launch_bounds__(256)
logmel_kernel(const float *__restrict__ power, const int *__restrict__ counts, int NBP, int M,
              int T_max, const aug::MelBin *melw, const int *melstart, float floor_v, float pad_v, int comp,
              float *__restrict__ feats) {
    extern __shared__ __align__(16) float sm[];
    float *fs = sm + logmel_fs(NBP);                                // [LM_FT][M | 1] band energies
    float4 *mw = reinterpret_cast<float4 *>(sm + logmel_mw(NBP, M));   // [NBP] (up, up, down, down)
    int *mst = reinterpret_cast<int *>(mw + NBP), *cut = mst + M + 2;
    // (the last utterances first: of power spectra made just now they are the ones still in L2)
    const int utt = gridDim.y - 1 - blockIdx.y, tid = threadIdx.x, ld = M | 1;
    const int t0 = blockIdx.x * LM_FT;
    const int rows = min(LM_FT, T_max - t0);
    const int T = min(max(counts[utt], 0), T_max);
    const int nf = max(0, min(rows, T - t0));
    // (the tables come from the kernel before; everything else was there when that one started)
    float *o = feats + ((int64_t)utt * T_max + t0) * M;
    fill_floats(o + nf * M, (rows - nf) * M, pad_v, tid, 256);
    if (nf == 0) {
        chain_wait();
        return;
    }
    const float *p = power + ((int64_t)utt * T_max + t0) * NBP;
    const int n = nf * NBP, shift = (int)((reinterpret_cast<uintptr_t>(p) >> 2) & 3);
    const int head = min(n, (4 - shift) & 3), n4 = (n - head) >> 2;
    float *pt = sm + shift;
    for (int i = tid; i < n4; i += 256)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         (unsigned)__cvta_generic_to_shared(pt + head + 4 * i)),
                     "l"(p + head + 4 * i)
                     : "memory");
    if (tid < head) pt[tid] = p[tid];
    const int tail = head + 4 * n4 + tid;
    if (tail < n) pt[tail] = p[tail];
    chain_wait();
    for (int k = tid; k < NBP; k += 256) {
        const aug::MelBin w = melw[(int64_t)utt * NBP + k];
        mw[k] = make_float4(w.up, w.up, w.down, w.down);
    }
    for (int m = tid; m < M + 2; m += 256) mst[m] = melstart[(int64_t)utt * (M + 2) + m];
    __syncthreads();
    cut_bands<LM_RUNS>(cut, mst, M, tid);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const int f = tid & 15, run = tid >> 4;          // frames f and f + 16 (its row may hold no frame)
    if (f < nf) {
        walk_bands(reinterpret_cast<const ulonglong2 *>(mw), mst, cut[run], cut[run + 1],
                   TwoRows{pt + f * NBP, f + 16 < nf ? 16 * NBP : 0}, fs + f * ld, 16 * ld);
    }
    __syncthreads();
    if ((M & 3) == 0 && (reinterpret_cast<uintptr_t>(feats) & 15) == 0) {
        const int m4 = M >> 2, step_f = 256 / m4, step_m = 256 - step_f * m4;
        int ff = tid / m4, m = tid - ff * m4;
        for (int i = tid; i < nf * m4; i += 256) {
            const float *e = fs + ff * ld + 4 * m;
            reinterpret_cast<float4 *>(o)[i] =
                make_float4(compress(e[0], floor_v, comp), compress(e[1], floor_v, comp),
                            compress(e[2], floor_v, comp), compress(e[3], floor_v, comp));
            ff += step_f;
            m += step_m;
            if (m >= m4) {
                m -= m4;
                ++ff;
            }
        }
    } else {
        for (int i = tid; i < nf * M; i += 256) {
            const int ff = i / M;
            o[i] = compress(fs[i + ff * (ld - M)], floor_v, comp);
        }
    }
}

template <int K, int MODE>
int launch_frames(AugCtx *ctx, const float *a, const float *b, int64_t stride, const int *lengths,
                  const AugUttParams *table, int B, float *out, int T_max, int *counts, int n_cap, float *wave = nullptr,
                  int64_t wave_stride = 0) {
    const AugConfig &c = ctx->cfg;
    constexpr int FT = tile_frames<K>(), RUN_TILES = Plan<K>::TILES;
    // Hops beyond several windows have a limit (AUG_ECAP), in samples of 32 (K = 1024: 8) frames that one
    // behind the other with their gaps fit a multiprocessor beside the tables.
    const int64_t reach = ((int64_t)(K == 512 ? 31 : 7) * c.hop + c.win + 3) & ~(int64_t)3;
    if (reach > (K == 1024 ? 43762 - c.n_mel : MODE == 0 ? 48736 : 47644 - ((c.n_mel + 5) & ~3))) return AUG_ECAP;
    // Copying one tile ahead needs rows that start on 16-byte boundaries, and room: where the buffers
    // for it do not fit (hops of 500 samples at K = 512, of 1000 at 1024) tiles are loaded when they are
    // needed, without the gaps where there are any (128 utterances of 10 s, K = 1024: hop 1000, window
    // 1024 394 us one sample after another, 276; hop 1600, window 800 538 and 240).
    Layout lay = make_layout<K, MODE>(c.win, c.hop, c.n_mel, AHEAD);
    if ((stride & 3) != 0 || sizeof(float) * lay.total > 227 * 1024)
        lay = make_layout<K, MODE>(c.win, c.hop, c.n_mel, packed_step(c.win, c.hop) < c.hop ? PACKED : DIRECT);
    const size_t smem = sizeof(float) * (size_t)lay.total;
    if (smem > 227 * 1024) return AUG_ECAP;
    // A CTA works through a run of tiles (window values, filterbank tables and other
    // set-up once per run) unless the batch is so small that single tiles are needed
    // to give every multiprocessor something to do.
    const int n_tiles = (T_max + FT - 1) / FT;
    const bool runs = (int64_t)n_tiles * B >= 2 * (int64_t)ctx->sm_count * RUN_TILES;
    const int n_runs = (n_tiles + RUN_TILES - 1) / RUN_TILES;
    RunMap map = {B, B, Divisor(n_runs), Divisor(n_tiles)};
    if (runs) map.long_utts = std::max(0, B - (TAIL_ROUNDS * 2 * ctx->sm_count + n_tiles - 1) / n_tiles);
    if (MODE == 0 && lay.ahead && lay.chunk_cap > TAIL_SAMPLES) {
        // Nothing copies the samples of single tiles ahead, and large ones of a power spectrum take twice as long for it: only
        // where that makes up for the last round of runs (100 utterances of 10 s: window and hop 320 51 us in runs
        // alone, 57 with single tiles at the end; window 512, hop 441 52 and 43).
        const int64_t places = 2 * (int64_t)ctx->sm_count, in_runs = (int64_t)map.long_utts * n_tiles;
        const int64_t alone = ((int64_t)n_runs * B + places - 1) / places * std::min(RUN_TILES, n_tiles);
        if ((in_runs + 2 * ((int64_t)B * n_tiles - in_runs)) / places + 2 > alone) map.long_utts = B;
    }
    const dim3 grid = runs ? dim3(map.long_utts * n_runs + (B - map.long_utts) * n_tiles) : dim3(n_tiles, B);
    auto kern = runs ? frames_kernel<K, MODE, RUN_TILES> : frames_kernel<K, MODE, 1>;
    if ((runs ? smem_opt_in<frames_kernel<K, MODE, RUN_TILES>>(ctx->device)
              : smem_opt_in<frames_kernel<K, MODE, 1>>(ctx->device)) != AUG_OK)
        return AUG_ECUDA;
    const GainSource gain = {nullptr, ctx->energy, table};
    // (MODE 0 reads what the caller's kernels wrote: launched the ordinary way)
    if (MODE == 1) {
        if (launch_chained(kern, grid, FEAT_THREADS, smem, ctx->stream, a, b, stride, gain, lengths, c.win, c.hop,
                           c.n_mel, T_max, ctx->melw, ctx->melstart, ctx->tw, c.log_floor, c.pad_value, c.compression,
                           out, counts, n_cap, wave, wave_stride, lay, map) != AUG_OK)
            return AUG_ECUDA;
    } else {
        kern<<<grid, FEAT_THREADS, smem, ctx->stream>>>(
            a, b, stride, gain, lengths, c.win, c.hop, c.n_mel, T_max, ctx->melw, ctx->melstart, ctx->tw,
            c.log_floor, c.pad_value, c.compression, out, counts, n_cap, wave, wave_stride, lay, map);
        AUG_CUDA_OK(cudaGetLastError());
    }
    ctx->launches++;
    return AUG_OK;
}

}  // namespace

int launch_mel_tables(AugCtx *ctx, const AugUttParams *table, int B, bool reset) {
    const AugConfig &c = ctx->cfg;
    const MelEdges e(c.f_lo, c.f_hi, c.n_mel);
    mel_tables_kernel<<<B, 256, 0, ctx->stream>>>(
        table, c.n_fft, c.n_mel, (double)c.fs, e.first, e.step, ctx->melw, ctx->melstart,
        c.vtlp_win > 0 ? 1 : 0, ctx->counters, reset ? ctx->energy : nullptr);
    AUG_CUDA_OK(cudaGetLastError());
    ctx->launches++;
    return AUG_OK;
}

int launch_stft_power(AugCtx *ctx, const float *wave, int64_t stride, const int *lengths, int B,
                      float *power, int T_max, int *counts) {
    if (T_max <= 0) return AUG_OK;
    const int n_cap = (int)(stride < 0x7fffffff ? stride : 0x7fffffff);     // the caller's rows end at their stride
    if (ctx->cfg.n_fft == 512)
        return launch_frames<512, 0>(ctx, wave, nullptr, stride, lengths, nullptr, B, power, T_max, counts, n_cap);
    return launch_frames<1024, 0>(ctx, wave, nullptr, stride, lengths, nullptr, B, power, T_max, counts, n_cap);
}

// max_len: the length clamp the convolution used, so that every stage cuts an over-long
// entry of `lengths` at the same sample.  wave (may be NULL): the mixed waveform is written on the
// way -- it is in shared memory anyway; a pass of its own over y_s and v took 33 us on 96
// utterances of 2-20 s -- unless frames leave gaps between them, or fewer feature rows than frames are
// asked for: what lies behind the last row is written by one CTA of the utterance (32 utterances of
// 20 s with one row 722 us, with a pass of its own 126).  A few frames more are let through,
// as without lengths on the host max_len is the row stride, which callers round up.
constexpr int WAVE_SLACK = 8;
bool features_write_wave(const AugCtx *ctx, int max_len, int T_max) {
    return ctx->cfg.hop <= ctx->cfg.win && frame_count(max_len, ctx->cfg.win, ctx->cfg.hop) <= (int64_t)T_max + WAVE_SLACK;
}
int launch_fused_features(AugCtx *ctx, const int *lengths, const AugUttParams *table, int B, float *feats, int T_max,
                          int *counts, int max_len, float *wave, int64_t wave_stride) {
    if (T_max <= 0) return AUG_OK;
    if (ctx->cfg.n_fft == 512)
        return launch_frames<512, 1>(ctx, ctx->ys, ctx->vv, ctx->ws_stride, lengths, table, B, feats, T_max, counts, max_len,
                                     wave, wave_stride);
    return launch_frames<1024, 1>(ctx, ctx->ys, ctx->vv, ctx->ws_stride, lengths, table, B, feats, T_max, counts, max_len,
                                  wave, wave_stride);
}

int launch_logmel(AugCtx *ctx, const float *power, const int *counts, int B, int T_max,
                  float *feats) {
    const AugConfig &c = ctx->cfg;
    if (T_max <= 0) return AUG_OK;
    const int NBP = ctx->n_bins;
    if (smem_opt_in<logmel_kernel>(ctx->device) != AUG_OK) return AUG_ECUDA;
    dim3 grid((T_max + LM_FT - 1) / LM_FT, B);
    if (launch_chained(logmel_kernel, grid, 256, logmel_smem(NBP, c.n_mel), ctx->stream, power, counts, NBP, c.n_mel,
                       T_max, ctx->melw, ctx->melstart, c.log_floor, c.pad_value, c.compression, feats) != AUG_OK)
        return AUG_ECUDA;
    ctx->launches++;
    return AUG_OK;
}

// ---------------------------------------------------------------- step 4 without any allocation
//
// feat_vtlp_logmel needs two small per-utterance tables (filterbank weights per
// DFT bin, first bin of every band interval) that normally live in the context's
// workspace, and a context cannot exist without cudaMalloc.  Some callers are not
// allowed to allocate: a plug-in running inside a host application that has
// handed every byte of device memory to its own pool, a real-time feature
// front-end that must not touch the allocator after start-up, or code that only
// receives device pointers and a stream.  For them the tables live in a
// fixed-size array that is part of the loaded library image, so nothing is
// allocated at call time -- at the price that every GPU that loads the library
// carries the array until the process exits, and that all calls share it.
namespace {

constexpr int NOALLOC_BINS = 513;                                   // n_fft <= 1024
constexpr size_t NOALLOC_MELW_BYTES =
    sizeof(aug::MelBin) * (size_t)AUG_NOALLOC_MAX_BATCH * NOALLOC_BINS;          // 1 050 624
constexpr size_t NOALLOC_START_BYTES =
    sizeof(int) * (size_t)AUG_NOALLOC_MAX_BATCH * (aug::MAX_MEL + 2);            //   133 120
static_assert(NOALLOC_MELW_BYTES % 256 == 0, "second table must stay 256-byte aligned");

// The scratch itself.  In host code this name is only a handle for the runtime,
// not an address a kernel could use; the device address is looked up below.
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_MELW_BYTES + NOALLOC_START_BYTES];

constexpr int NOALLOC_MAX_DEVICES = 64;
void *g_noalloc_addr[NOALLOC_MAX_DEVICES];   // device address of the scratch, per device; NULL = not looked up yet

// Device address of the scratch on the current device.  The first call on a
// device asks the runtime for it (no allocation: the array already exists in the
// module); later calls reuse the cached pointer.
int noalloc_scratch(void **out) {
    int dev = -1;
    AUG_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return AUG_ECAP;
    void *p = __atomic_load_n(&g_noalloc_addr[dev], __ATOMIC_ACQUIRE);
    if (!p) {
        AUG_CUDA_OK(cudaGetSymbolAddress(&p, g_noalloc_scratch));
        if (!p) return AUG_ECUDA;
        __atomic_store_n(&g_noalloc_addr[dev], p, __ATOMIC_RELEASE);   // same value from any thread
    }
    *out = p;
    return AUG_OK;
}

}  // namespace

extern "C" int feat_vtlp_logmel_noalloc(const AugConfig *cfg, const float *power_dev,
                                        const int *frame_counts_dev,
                                        const AugUttParams *table_dev, int B, int T_max,
                                        float *feats_dev, void *cuda_stream) {
    if (!cfg || !power_dev || !frame_counts_dev || !table_dev || !feats_dev) return AUG_EINVAL;
    if (B < 0 || T_max <= 0) return AUG_EINVAL;
    if (cfg->n_fft != 512 && cfg->n_fft != 1024) return AUG_EINVAL;
    if (cfg->n_mel < 1 || cfg->fs <= 0 || !(cfg->f_lo >= 0.f) || !(cfg->f_hi > cfg->f_lo) ||
        cfg->f_hi > 0.5f * cfg->fs + 1e-3f || !(cfg->log_floor > 0.f) || !isfinite(cfg->pad_value))
        return AUG_EINVAL;
    if (cfg->compression != AUG_COMPRESS_LOG && cfg->compression != AUG_COMPRESS_POW_1_15)
        return AUG_EINVAL;
    // the fixed scratch holds tables for this many utterances and bands, no more
    if (B > AUG_NOALLOC_MAX_BATCH || cfg->n_mel > aug::MAX_MEL) return AUG_ECAP;
    if (B == 0) return AUG_OK;

    void *scratch = nullptr;
    int rc = noalloc_scratch(&scratch);
    if (rc != AUG_OK) return rc;
    aug::MelBin *melw = reinterpret_cast<aug::MelBin *>(scratch);
    int *melstart = reinterpret_cast<int *>(static_cast<unsigned char *>(scratch) + NOALLOC_MELW_BYTES);

    // Both tables are written in full for utterances [0, B) before they are read
    // (same stream), so nothing left by an earlier call is ever seen and nothing
    // needs clearing.
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int nbp = cfg->n_fft / 2 + 1;
    const MelEdges e(cfg->f_lo, cfg->f_hi, cfg->n_mel);
    mel_tables_kernel<<<B, 256, 0, st>>>(table_dev, cfg->n_fft, cfg->n_mel, (double)cfg->fs, e.first, e.step, melw,
                                         melstart, 0, nullptr, nullptr);
    AUG_CUDA_OK(cudaGetLastError());
    int dev = -1;
    AUG_CUDA_OK(cudaGetDevice(&dev));
    if (smem_opt_in<logmel_kernel>(dev) != AUG_OK) return AUG_ECUDA;
    dim3 grid((T_max + LM_FT - 1) / LM_FT, B);
    logmel_kernel<<<grid, 256, logmel_smem(nbp, cfg->n_mel), st>>>(power_dev, frame_counts_dev, nbp, cfg->n_mel, T_max,
                                           melw, melstart, cfg->log_floor, cfg->pad_value,
                                           cfg->compression, feats_dev);
    AUG_CUDA_OK(cudaGetLastError());
    return AUG_OK;
}
