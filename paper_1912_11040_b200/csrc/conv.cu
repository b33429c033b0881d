// Step 2: reverberation by FFT overlap convolution, noise mixing.
//
// Every route is overlap-save in form: an output block is computed from the input
// segment that ends with it (the block plus the samples before it that the response
// reaches back to), which is the overlap-add tail sum moved to the input side, so
// output blocks never exchange data.  All transforms are real ones of 16384 points
// (fft_pair.cuh).  The route is fixed by the response length:
//
//   up to 8192 taps   ONE partition, 16384 - taps + 1 outputs per block: a block of one output is
//                     done in one go -- forward, multiply, inverse -- and nothing but y_s and v
//                     is stored.  Several noise sources are summed in the frequency domain
//                     through a small parking area in global memory (one inverse).
//   longer            partitions of 8192 taps, blocks of 8192 outputs, Y_b = sum_p X_{b-p} H_p with
//                     X_j the spectrum of the 16384 samples that end with block j: every X_j is
//                     stored once; the spectra a block needs are read back (mostly from L2),
//                     multiplied and accumulated in registers -- all noise sources in one sum --
//                     and inverse-transformed.  On 128 x 8 s with 24000 taps and three noises
//                     this takes 488 us; 4096-tap partitions of 8192-point scalar transforms,
//                     twice the products per sample and twice the bytes from L2, took 534.
//
// Responses are often shorter than their buffer: behind the last image source's window
// every tap is exactly zero.  The number of taps up to the last non-zero one (the largest over an utterance's
// sources) is recorded where the responses are made; those of the caller are measured, by a kernel of their own or
// by the one that transforms them.  The fused route then takes 16384 - that + 1 outputs from every block
// instead of 16384 - rir_taps + 1, and the stored-spectra route skips the partitions
// that are zero throughout.  A context sized for long responses sends a batch whose
// responses all end within 8192 taps through the fused route as well: the kernels of
// both routes are launched, look at the batch's largest effective length first, and
// those of the route not taken return at once.  The largest effective length of a batch
// is also copied to the host without waiting for it; while the last value seen says
// "long", the next call launches the stored-spectra kernels alone (they serve any
// length), so a stream of long-response batches pays nothing for the choice.  (Routing
// utterance by utterance was
// measured too: a minority of long CTAs of the fused kernel beside the stored-spectra
// kernels balanced badly.)  The result is the same convolution.
#include <algorithm>

#include "common.cuh"
#include "fft_pair.cuh"

namespace {

constexpr int CT = 256;                // threads per CTA of the smaller kernels
constexpr int FUSED_MINB = 2;          // CTAs per SM of the transforming kernels

// Source s of an utterance: pointer to its samples, loop length; false if the row's
// noise stretch is unusable (reported once through the status word).
__device__ __forceinline__ bool source_of(const AugUttParams &row, int s, const float *speech_row,
                                          const float *bank, int64_t bank_len, const float *&x,
                                          int &nlen) {
    if (s == 0) {
        x = speech_row;
        nlen = 1;
        return true;
    }
    const int64_t off = row.noise_offset[s - 1];
    nlen = row.noise_len[s - 1];
    if (nlen <= 0 || off < 0 || off + nlen > bank_len || bank == nullptr) return false;
    x = bank + off;
    return true;
}

// Effective length of the responses: (index + 1) of the last non-zero tap (leff[utt][source]), and the largest of
// the batch (*leff_all, zeroed before the launch).  For responses that come from the caller.
__global__ void __launch_bounds__(CT)
rir_length_kernel(const float *rir, const AugUttParams *__restrict__ table, int S_max, int L,
                  int *__restrict__ leff, int *__restrict__ leff_all) {
    __shared__ int red_i[CT / 32];
    const int s = blockIdx.x, utt = blockIdx.y, t = threadIdx.x;
    chain_next();
    chain_wait();
    const AugUttParams &row = table[utt];
    if (row.n_src < 1 || row.n_src > S_max || s >= row.n_src) return;
    const float *h = rir + ((int64_t)utt * S_max + s) * L;
    int last = 0;
    if ((reinterpret_cast<uintptr_t>(h) & 15) == 0) {
        for (int i = 4 * t; i + 3 < L; i += 4 * CT) {
            const float4 z = *reinterpret_cast<const float4 *>(h + i);
            if (z.x != 0.f) last = i + 1;
            if (z.y != 0.f) last = i + 2;
            if (z.z != 0.f) last = i + 3;
            if (z.w != 0.f) last = i + 4;
        }
        for (int i = (L & ~3) + t; i < L; i += CT)
            if (h[i] != 0.f) last = max(last, i + 1);
    } else {
        for (int i = t; i < L; i += CT)
            if (h[i] != 0.f) last = i + 1;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
    if ((t & 31) == 0) red_i[t >> 5] = last;
    __syncthreads();
    if (t == 0) {
        int m = 0;
        for (int i = 0; i < CT / 32; ++i) m = max(m, red_i[i]);
        leff[utt * S_max + s] = m;
        if (m > 0) atomicMax(leff_all, m);
    }
}

// Which route a batch takes in a context sized for responses of more than 8192 taps.
__device__ __forceinline__ bool takes_fused_route(int leff_batch) { return leff_batch <= aug::CONV_TAPS; }

// ---------------------------------------------------------------- mixing
// The gain once per utterance, ahead of the mix of aug_reverb_mix; the feature kernel works it out while its first
// samples are on their way, and so does the mix of aug_pipeline (every thread of it, under its loads: 32 utterances of
// 20 s with the waveform and one feature row 132.4 us with this launch ahead of the mix, 131.8 without, 256 of 10 s 450 and
// 448; by one thread of a CTA for all 128.7 and 422.6 where by every one 129.1 and 422.0).
__global__ void __launch_bounds__(256)
snr_gain_kernel(const double *energy, const AugUttParams *__restrict__ table, int B,
                float *__restrict__ gain) {
    const int utt = blockIdx.x * 256 + threadIdx.x;
    const double ratio = utt < B ? snr_ratio(table[utt]) : 1.0;
    chain_next();
    chain_wait();
    if (utt < B) gain[utt] = snr_gain(energy[2 * utt], energy[2 * utt + 1], ratio, table[utt].n_src);
}

// A pass over y_s and v, bound by memory: 4096 samples per CTA, eight 128-bit loads in flight per
// thread.
// READY: the gain has been worked out.  (Without the fp64 arithmetic 48 registers instead of 64, and 12.5 us instead
// of 13.2 for 64 utterances of 5-10 s.)
constexpr int MIX_GROUPS = 4;              // 128-bit groups per thread
template <bool READY>
__global__ void __launch_bounds__(256)
mix_kernel(const float *ys, const float *vv, int64_t ws_stride,
           const GainSource gain, const int *__restrict__ lengths,
           float *__restrict__ out, int64_t out_stride, int n_cap) {
    const int utt = blockIdx.y, tid = threadIdx.x;
    chain_wait();
    const int N = min(max(lengths[utt], 0), n_cap);
    const int i0 = blockIdx.x * (MIX_GROUPS * 1024) + 4 * tid;
    if (blockIdx.x * (MIX_GROUPS * 1024) >= N) return;
    const float *a = ys + (int64_t)utt * ws_stride;
    const float *b = vv + (int64_t)utt * ws_stride;
    float *o = out + (int64_t)utt * out_stride;
    float4 x[MIX_GROUPS], y[MIX_GROUPS];
#pragma unroll
    for (int u = 0; u < MIX_GROUPS; ++u) {
        const int i = i0 + 1024 * u;           // (workspace rows are allocated up to a multiple of 4)
        if (i < N) {
            x[u] = *reinterpret_cast<const float4 *>(a + i);
            y[u] = *reinterpret_cast<const float4 *>(b + i);
        }
    }
    const float g = fabsf(READY ? gain.value[utt]
                                : snr_gain(gain.energy[2 * utt], gain.energy[2 * utt + 1], snr_ratio(gain.table[utt]),
                                           gain.table[utt].n_src));
#pragma unroll
    for (int u = 0; u < MIX_GROUPS; ++u) {
        const int i = i0 + 1024 * u;
        const float4 z = make_float4(fmaf(g, y[u].x, x[u].x), fmaf(g, y[u].y, x[u].y), fmaf(g, y[u].z, x[u].z),
                                     fmaf(g, y[u].w, x[u].w));
        if (i + 3 < N) {
            *reinterpret_cast<float4 *>(o + i) = z;
        } else if (i < N) {
            o[i] = z.x;
            if (i + 1 < N) o[i + 1] = z.y;
            if (i + 2 < N) o[i + 2] = z.z;
        }
    }
}

// ================================================================ 8192-sample blocks
// Impulse responses of up to 8192 taps fit one partition of a 16384-point real
// transform, so a CTA can do a whole block of one output -- forward, multiply, inverse --
// without any stored spectra.  The even and the odd samples of a segment are two real
// sequences of 8192 points, each a complex transform of 4096 points on pairs of its
// samples: four consecutive samples x0..x3 are one point of both, (x0, x1) their real and
// (x2, x3) their imaginary parts, which is the layout the packed arithmetic of
// fft_pair.cuh wants.  After the forward transform thread t holds, for r < 8, the
// frequencies k = j + 256 r and (from its partner lane) 4096 - k of both; from these it forms
// the bins k, 8192-k, 4096-k and 4096+k of the segment's spectrum, multiplies them with the
// response's and folds the products back, all in registers.  The response's spectra are
// stored in the order the threads read them.
constexpr int BLK2 = aug::CONV_TAPS;   // most taps of a partition
constexpr int F2 = 2 * BLK2;           // real transform size
constexpr int NB2 = F2 / 2;            // complex numbers stored per spectrum
constexpr int CF = fftpair::THREADS;   // threads per CTA
constexpr int NP2 = 4096 / CF;         // points per thread
constexpr int NS2 = NP2 / 2;           // slots (k, 4096-k) per thread
using fftpair::C2;
using fftpair::u64;

// Asynchronous copy global -> shared; `bytes` are read, the rest is zero.
__device__ __forceinline__ void copy4_async(float *dst_smem, const float *src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst_smem)),
                 "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// F2 input samples starting at `base`: thread t gets samples base + 4 (t + 256 r) + {0, 1} and
// + {2, 3} as the real and imaginary parts of point r.  Speech reads x[i]; a noise source
// reads its stretch of the bank end to end (x[i mod nlen]).  Outside [0, N): zero.  The
// exchange buffer must be free.  (Nobody writes the audio while this kernel lives: it is the caller's, or
// the warped speech, whose kernel lets none start beside it.)
__device__ __forceinline__ void load_segment(C2 *v, fftpair::Shared &sh, const float *__restrict__ x, bool looped,
                                             int nlen, int base, int N, int t) {
    // A segment that lies inside the utterance (most do), and for a looped stretch inside one
    // period of it, is read straight into registers: the same for the whole CTA.
    if (base >= 0 && base + F2 <= N) {
        const int m0 = looped ? base % nlen : base;
        if (!looped || m0 + F2 <= nlen) {
            const float *p = x + m0 + 4 * t;
            if ((reinterpret_cast<uintptr_t>(p) & 15) == 0) {
#pragma unroll
                for (int r = 0; r < NP2; ++r)
                    asm("ld.global.nc.L1::no_allocate.v2.u64 {%0, %1}, [%2];"
                        : "=l"(v[r].re), "=l"(v[r].im)
                        : "l"(p + 4 * CF * r));
            } else {
                // any other offset: single words, which the four loads of a group share in L1
#pragma unroll
                for (int r = 0; r < NP2; ++r) {
                    const float *q = p + 4 * CF * r;
                    v[r] = {fftpair::pack(__ldg(q), __ldg(q + 1)), fftpair::pack(__ldg(q + 2), __ldg(q + 3))};
                }
            }
            return;
        }
    }
    if (!looped || ((nlen & 3) == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0)) {
        // groups of four lie on 16-byte boundaries and never wrap; rows and stretches hold whole groups
        int i = base + 4 * t, m = i, step = 4 * CF, wrap = 0x7fffffff;
        if (looped) {
            m = i >= 0 ? i % nlen : (nlen - (-i) % nlen) % nlen;
            step %= nlen;
            wrap = nlen;
        }
#pragma unroll
        for (int r = 0; r < NP2; ++r) {
            float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            if ((unsigned)i < (unsigned)N) z = __ldg(reinterpret_cast<const float4 *>(x + m));
            v[r] = {fftpair::pack(z.x, i + 1 < N ? z.y : 0.f),
                    fftpair::pack(i + 2 < N ? z.z : 0.f, i + 3 < N ? z.w : 0.f)};
            i += 4 * CF;
            m += step;
            if (m >= wrap) m -= wrap;
        }
        return;
    }
    // sample by sample through the exchange buffer, neighbouring threads neighbouring samples
    {
        __syncthreads();
        int i = base + t, m = i >= 0 ? i % nlen : (nlen - (-i) % nlen) % nlen;
        const int step = CF % nlen;
        float *dst = reinterpret_cast<float *>((t & 2 ? sh.im : sh.re) + fftpair::slot(t >> 2)) + (t & 1);
#pragma unroll 4
        for (int r = 0; r < F2 / CF; ++r) {
            copy4_async(dst, x + m, (unsigned)i < (unsigned)N ? 4 : 0);
            dst += 2 * fftpair::slot(CF / 4);
            i += CF;
            m += step;
            if (m >= nlen) m -= nlen;
        }
        copies_done();
        __syncthreads();
    }
    fftpair::load16<fftpair::slot(CF)>(v, sh, fftpair::slot(t));
}

// The four bins a thread forms from frequencies k and m = 4096-k of the two half
// transforms, lanes (k, m):  p = X[k], conj X[m];  q = conj X[8192-k], X[4096+k].
// Thread j = 0 has in its first slot the frequencies 0 and 2048 instead:
// p = (X[0], Re X[4096]; X[8192], Im X[4096]), q = (X[2048], conj X[6144]).
// All are twice the value of the transform (the factor sits in the stored responses).
struct Bins {
    u64 pr, pi, qr, qi;
};
__device__ __forceinline__ u64 low2(u64 a, u64 b) { return fftpair::pack(fftpair::unpack(a).x, fftpair::unpack(b).x); }
__device__ __forceinline__ u64 high2(u64 a, u64 b) { return fftpair::pack(fftpair::unpack(a).y, fftpair::unpack(b).y); }

// U = exp(-2 pi i k / 16384) of slot r and, by squaring, W = exp(-2 pi i k / 8192), from
// u = exp(-2 pi i j / 16384), k = j + 256 r
struct SplitTwiddle {
    u64 ur, ui;            // lanes (U^k, conj U^m), conj U^m = i U^k
    u64 wx, wy;
    __device__ __forceinline__ SplitTwiddle(float2 u, int r) {
        using namespace fftpair;
        // exp(-i pi r / 32)
        const float cr[8] = {1.f, 0.99518472667219688624f, 0.98078528040323044913f, 0.95694033573220886494f,
                             0.92387953251128675613f, 0.88192126434835502971f, 0.83146961230254523708f,
                             0.77301045336273696081f};
        const float ci[8] = {0.f, -0.09801714032956060199f, -0.19509032201612826785f, -0.29028467725446236764f,
                             -0.38268343236508977173f, -0.47139673682599764856f, -0.55557023301960222474f,
                             -0.63439328416364549822f};
        const float x = r ? fmaf(u.x, cr[r], -u.y * ci[r]) : u.x, y = r ? fmaf(u.x, ci[r], u.y * cr[r]) : u.y;
        ur = pack(x, -y);
        ui = pack(y, x);
        const float p = fmaf(x, x, -y * y), q = 2.f * x * y;
        wx = both(p);
        wy = both(q);
    }
};
// Spectra E, O of the even and odd samples at k and (conjugated) at m = 4096-k; then
// X = E +- U^k O in lanes (X[k], conj X[m]).
__device__ __forceinline__ Bins bins_forward(C2 zk, C2 zm, const SplitTwiddle &w) {
    using namespace fftpair;
    const u64 evr = add2(zk.re, zm.re), evi = sub2(zk.im, zm.im);
    const u64 odr = add2(zk.im, zm.im), nodi = sub2(zk.re, zm.re);
    const u64 wor = fma2(w.wy, nodi, mul2(w.wx, odr));
    const u64 nwoi = sub2(mul2(w.wx, nodi), mul2(w.wy, odr));
    const C2 ek = {add2(evr, wor), sub2(evi, nwoi)}, em = {sub2(evr, wor), add2(evi, nwoi)};
    // lanes from (even, odd) to (k, m)
    const u64 er = low2(ek.re, em.re), ei = low2(ek.im, em.im);
    const u64 orr = high2(ek.re, em.re), oi = high2(ek.im, em.im);
    const u64 tr = sub2(mul2(w.ur, orr), mul2(w.ui, oi)), ti = fma2(w.ui, orr, mul2(w.ur, oi));
    return {add2(er, tr), add2(ei, ti), sub2(er, tr), sub2(ei, ti)};
}
// Products back to the frequencies of the two half-size transforms (again twice the value),
// real and imaginary parts swapped for the inverse.
__device__ __forceinline__ void bins_inverse(const Bins &y, const SplitTwiddle &w, C2 &zk, C2 &zm) {
    using namespace fftpair;
    const u64 er = add2(y.pr, y.qr), ei = add2(y.pi, y.qi);
    const u64 dr = sub2(y.pr, y.qr), di = sub2(y.pi, y.qi);
    const u64 orr = fma2(w.ui, di, mul2(w.ur, dr)), oi = sub2(mul2(w.ur, di), mul2(w.ui, dr));
    // lanes from (k, m) to (even, odd)
    const u64 ekr = low2(er, orr), emr = high2(er, orr), eki = low2(ei, oi), emi = high2(ei, oi);
    const u64 ar = add2(ekr, emr), ai = add2(eki, emi);           // Ek + conj Em
    const u64 cr = sub2(ekr, emr), ci = sub2(eki, emi);           // Ek - conj Em
    // i conj(W) c, its real part with the other sign
    const u64 nqr = sub2(mul2(w.wx, ci), mul2(w.wy, cr)), qi = fma2(w.wy, ci, mul2(w.wx, cr));
    zk = {add2(ai, qi), sub2(ar, nqr)};
    zm = {sub2(qi, ai), add2(ar, nqr)};
}
__device__ __forceinline__ Bins edge_forward(C2 z0, C2 zh) {
    using namespace fftpair;
    const float h = 0.70710678118654752440f;                      // U^2048 = (h, -h)
    const float2 r = unpack(z0.re), i = unpack(z0.im), hr = unpack(zh.re), hi = unpack(zh.im);
    const float e0 = 2.f * (r.x + i.x), e4 = 2.f * (r.x - i.x), o0 = 2.f * (r.y + i.y), o4 = 2.f * (r.y - i.y);
    const float er = 2.f * hr.x, ei = -2.f * hi.x, orr = 2.f * hr.y, oi = -2.f * hi.y;
    const float tr = h * (orr + oi), ti = h * (oi - orr);
    return {pack(e0 + o0, e4), pack(e0 - o0, -o4), pack(er + tr, er - tr), pack(ei + ti, ei - ti)};
}
__device__ __forceinline__ void edge_inverse(const Bins &y, C2 &z0, C2 &zh) {
    using namespace fftpair;
    const float h = 0.70710678118654752440f;
    const float2 pr = unpack(y.pr), pi = unpack(y.pi), qr = unpack(y.qr), qi = unpack(y.qi);
    const float e0 = pr.x + pi.x, o0 = pr.x - pi.x, e4 = 2.f * pr.y, o4 = -2.f * pi.y;
    z0 = {pack(e0 - e4, o0 - o4), pack(e0 + e4, o0 + o4)};
    const float er = qr.x + qr.y, ei = qi.x + qi.y, dr = qr.x - qr.y, di = qi.x - qi.y;
    const float orr = h * (dr - di), oi = h * (di + dr);
    zh = {pack(-2.f * ei, -2.f * oi), pack(2.f * er, 2.f * orr)};
}
__device__ __forceinline__ void multiply(u64 &xr, u64 &xi, u64 hr, u64 hi) {
    using namespace fftpair;
    const u64 yr = sub2(mul2(xr, hr), mul2(xi, hi));
    xi = fma2(xi, hr, mul2(xr, hi));
    xr = yr;
}
__device__ __forceinline__ void edge_multiply(Bins &y, const Bins &h) {
    using namespace fftpair;
    const float2 pr = unpack(y.pr), pi = unpack(y.pi), hr = unpack(h.pr), hi = unpack(h.pi);
    y.pr = pack(pr.x * hr.x, pr.y * hr.y - pi.y * hi.y);
    y.pi = pack(pi.x * hi.x, pr.y * hi.y + pi.y * hr.y);
    multiply(y.qr, y.qi, h.qr, h.qi);
}
// Bins of a slot of thread t at p + t, the halves CF apart; streamed, not kept in L1.  (The address follows
// from the plan, which is read behind chain_wait().)
__device__ __forceinline__ Bins load_bins(const float4 *p) {
    Bins z;
    asm("ld.global.L1::no_allocate.v2.u64 {%0, %1}, [%2];" : "=l"(z.pr), "=l"(z.pi) : "l"(p));
    asm("ld.global.L1::no_allocate.v2.u64 {%0, %1}, [%2];" : "=l"(z.qr), "=l"(z.qi) : "l"(p + CF));
    return z;
}
// A whole spectrum into L2, by one thread.
__device__ __forceinline__ void prefetch_spectrum(const float4 *p) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "n"(8 * NB2) : "memory");
}
__device__ __forceinline__ Bins load_parked(const float4 *p) {
    const ulonglong2 a = __ldcg(reinterpret_cast<const ulonglong2 *>(p));
    const ulonglong2 b = __ldcg(reinterpret_cast<const ulonglong2 *>(p + CF));
    return {a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ void store_bins(float4 *p, const Bins &z) {
    __stcg(reinterpret_cast<ulonglong2 *>(p), make_ulonglong2(z.pr, z.pi));
    __stcg(reinterpret_cast<ulonglong2 *>(p + CF), make_ulonglong2(z.qr, z.qi));
}

// ---------------------------------------------------------------- the list of work
// One unit of work is one block of one output (the reverberant speech, or the sum of the noise
// sources) of an utterance.  plan_kernel lists the units that exist -- how many blocks an
// utterance has depends on its length and on where its responses end -- and what they need to
// know; the convolving kernels' CTAs, as many as fit the device, work through the list.  With one CTA
// per possible block instead, 55 of 527 us (256 utterances of 2-20 s) went to launching CTAs
// (two thirds of them without work) and to each one's chain of loads before its first sample.
//
// Sums of several noise sources are the heavy units (three transforms and more against two), and blocks of noise that may
// have copies to write (below) come after them.  There are three lists, drawn from in this order: sums from the front,
// blocks with copies behind the others' room, the others from the back, so that no long unit is the last that the
// device waits for (in the order in which they are planned, and sums first: 64 utterances of 2-16 s, one or two noises,
// 167 and 153 us; 96 of 2-20 s with up to two 302 and 287; 256 of 2-20 s 720 and 706; 64 of 60 s with two 1409 and 1376,
// whole calls each.  Blocks with copies among the others, among the sums and between them: 64 of 2-16 s with recorded
// responses 150.8, 152.8 and 149.2; 96 of 2-20 s 272.6, 269.8 and 268.6; 4096 of 1-6 s 3276, 3273 and 3256).
//
// A stretch of noise that is shorter than the utterance repeats, and so does its reverberation as soon as the
// response has run in: v[n + P] = v[n], n >= taps - 1.  Where there is one noise source, only the blocks
// up to P + taps - 1 are listed, and those that hold the last period also write it wherever it comes back (4096
// utterances of 1-6 s, stretches of half to all of their length: 3365 us a call without copies, 3267 with them).
// P is a multiple of the stretch that leaves MOST_COPIES copies of a block at most, so that the writing is shared
// out: 64 utterances of 60 s over stretches of 1 s 782 us without copies, 666 with one period and all the others
// in a few CTAs' hands, 651 with three copies, 629 with seven; of 16001 samples 814, 972, 669 and 640.  Contexts for
// batches of less than two rounds of CTAs compute all blocks, see plan_args.
constexpr int MOST_COPIES = 7;
struct Plan {
    const float *x[AUG_S_MAX];     // [0] speech row, [1..n_noise] usable stretches of the bank
    int nlen[AUG_S_MAX];           // their lengths ([0] unused)
    int src[AUG_S_MAX];            // their source numbers
    int n_src;                     // 0: the row was rejected, both outputs are silence
    int n_noise;
    int N;                         // samples of the utterance
    int ob;                        // outputs per block
    int parts;                     // partitions that are not zero throughout (stored-spectra route)
    int period, copy_from;         // v from copy_from on comes back every `period` samples up to the end (0: it is computed)
};
struct Unit {
    int utt;
    int block2;                    // 2 block + (1 for the noise sum)
};
static_assert(sizeof(Plan) % 4 == 0 && sizeof(Plan) <= aug::PLAN_BYTES && sizeof(Unit) == 8, "");

// All that planning an utterance takes; n_cap: rows are not read beyond.
struct PlanArgs {
    const float *speech;
    int64_t stride;
    const int *lengths;
    const float *bank;
    int64_t bank_len;
    int n_cap;
    int *status;
    Plan *plans;
    Unit *units;
    int unit_cap;
    int *counters;                 // [N_COUNTERS]
    int repeats;                   // blocks of repeated noise are copied, not computed
};
// What planning reads of the caller's inputs: lane l the length of the utterance and source l (0: the speech) of its row.
// (Read, where the responses are made by the kernel before, ahead of the wait for it.)
struct PlanInput {
    int N, n_src;                  // n_src 0: the row was rejected (reported by step 1)
    const float *x;                // NULL: the stretch is unusable
    int nlen;
};
__device__ __forceinline__ PlanInput plan_input(const PlanArgs &a, const AugUttParams &row, int utt, int S_max, int lane) {
    PlanInput in;
    in.N = min(max(a.lengths[utt], 0), a.n_cap);
    in.n_src = row.n_src >= 1 && row.n_src <= S_max ? row.n_src : 0;
    in.x = nullptr;
    in.nlen = 0;
    if (lane < max(in.n_src, 1) && !source_of(row, lane, a.speech + (int64_t)utt * a.stride, a.bank, a.bank_len, in.x, in.nlen))
        in.x = nullptr;
    return in;
}
// By one warp; leff: taps up to the last non-zero one.
__device__ __forceinline__ void plan_utterance(const PlanArgs &a, const PlanInput &in, int utt, int leff, bool stored, int lane) {
    const int N = in.N;
    // every block yields the F2 - (taps - 1) outputs that see no wrap-around, cut to a multiple
    // of 4, where taps counts up to the last non-zero tap of this utterance's responses
    const int ob = stored ? BLK2 : (F2 - min(max(leff, 1), BLK2) + 1) & ~3;
    const int n = (N + ob - 1) / ob;
    // usable noises in the order of the sources
    const unsigned usable = __ballot_sync(0xffffffffu, lane > 0 && lane < in.n_src && in.x != nullptr);
    const int n_noise = __popc(usable), nlen = __shfl_sync(0xffffffffu, in.nlen, __ffs(usable | 0x80000000u) - 1);
    if (lane > 0 && lane < in.n_src && in.x == nullptr && n > 0 && atomicCAS(&a.status[0], -1, utt) == -1)
        a.status[1] = aug::R_NOISE;
    int n_v = n, period = 0;                       // blocks of v
    if (a.repeats && !stored && n_noise == 1 && nlen < N) {
        // as many stretches as keep the copies of a block few, and none shorter than a block
        const unsigned least = max(ob, (N - 1) / (MOST_COPIES + 1) + 1), one = max(nlen, 1);
        const unsigned several = (least + one - 1) / one * one;
        const unsigned blocks = several < (unsigned)N ? (several + (unsigned)max(leff, 1) - 2u) / (unsigned)ob + 1 : n;
        if ((int)blocks < n) {
            n_v = blocks;
            period = several;
        }
    }
    Plan *p = a.plans + utt;
    if (lane == 0 || (usable >> lane & 1)) {
        const int at = lane == 0 ? 0 : 1 + __popc(usable & ((1u << lane) - 1u));
        p->x[at] = in.x;
        p->nlen[at] = in.nlen;
        p->src[at] = lane;
    }
    int at = 0, at_v = 0;
    const bool heavy = n_noise > 1, copies = period > 0;
    if (lane == 0) {
        if (n > 0) {
            int *list = a.counters + (stored ? aug::LIST_STORED : aug::LIST_FUSED);
            if (heavy || copies) at_v = atomicAdd(list + (heavy ? 0 : 1), n_v);
            at = atomicAdd(list + 2, heavy || copies ? n : n + n_v);
        }
        p->n_src = in.n_src;
        p->n_noise = n_noise;
        p->N = N;
        p->ob = ob;
        p->parts = (max(leff, 1) + BLK2 - 1) / BLK2;
        p->period = period;
        p->copy_from = n_v * ob - period;
    }
    at = __shfl_sync(0xffffffffu, at, 0);
    at_v = __shfl_sync(0xffffffffu, at_v, 0);
    const int last = a.unit_cap - 1;
    for (int i = lane; i < n; i += 32) {
        a.units[last - at - i] = Unit{utt, 2 * i};
        if (i < n_v) a.units[heavy ? at_v + i : copies ? a.unit_cap + at_v + i : last - at - n - i] = Unit{utt, 2 * i + 1};
    }
}

// Largest length of an utterance's responses.
__device__ __forceinline__ int longest(const int *leff, const PlanInput &in, int utt, int S_max, int lane) {
    return __reduce_max_sync(0xffffffffu, lane < in.n_src ? leff[utt * S_max + lane] : 0);
}
// One warp per utterance (long responses of the caller: the route follows from the whole batch; elsewhere
// rir_spectra2_kernel plans on the way).
__global__ void __launch_bounds__(256)
plan_kernel(const __grid_constant__ PlanArgs args, const AugUttParams *__restrict__ table, int B, int S_max,
            const int *leff, const int *leff_all, int stored_only) {
    const int utt = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    PlanInput in;
    if (utt < B) in = plan_input(args, table[utt], utt, S_max, lane);
    chain_wait();
    // (not before: the next kernel's CTAs would wait in places that the responses' transforms still need.  aug_reverb_mix, 8
    // utterances of 5 s, three noises, responses of 24000 taps 73 us, so 62; of 12000 67 and 60)
    chain_next();
    if (utt < B)
        plan_utterance(args, in, utt, longest(leff, in, utt, S_max, lane), stored_only || !takes_fused_route(*leff_all), lane);
}

// Spectra of the partitions of each impulse response: 8192 taps (those beyond L are zero) and as many
// zeros, scaled by the noise weight and 1/F (and by 1/4 for
// the two doubled spectra of a product).  A chain of short loads, a transform and a store of 64 KB;
// the taps are requested together, four a load (256 x 3 responses of 8192 taps: 31.1 us one
// by one, 29.9; a test per group inside the loop parts the loads: 33.6).  Persistent CTAs that work
// through the partitions, as the kernels below, took 33.2 and, 128 x 4 x 3 partitions, 53 against 43.
//
// LENGTHS  KNOWN  where the responses end has been recorded: zeros behind are not read, partitions of zeros left out
//          FIND   responses of the caller, of one partition: found on the way.  The CTA that adds an utterance's last
//                 source plans its work; the sum it learns that from holds the lengths too and is asked for before
//                 the transform, read behind it
// The first n_plan CTAs plan instead (KNOWN: the kernel that made the responses measured them), a warp an
// utterance.  With a chain of atomics and the plan of the utterance ahead of the transform, 4096 x 2 responses
// of 4096 taps took 267 us, so 207.
enum Lengths { KNOWN, FIND };
template <Lengths LENGTHS>
__global__ void __launch_bounds__(CF, FUSED_MINB)
rir_spectra2_kernel(const float *rir, const AugUttParams *__restrict__ table, int B, int S_max,
                    int L, int P, const float2 *__restrict__ tw, float4 *__restrict__ hspec, const int *leff,
                    unsigned long long *arrived, const __grid_constant__ PlanArgs plan, int n_plan, const int *leff_all,
                    int mixed, int stored_only) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fftpair::Shared &sh = *reinterpret_cast<fftpair::Shared *>(smem_raw);
    __shared__ int red_i[CF / 32];
    const int t = threadIdx.x;
    if (LENGTHS == KNOWN && blockIdx.x < n_plan) {
        const int utt = blockIdx.x * (CF / 32) + (t >> 5), lane = t & 31;
        PlanInput in;
        if (utt < B) in = plan_input(plan, table[utt], utt, S_max, lane);
        chain_wait();
        if (utt < B)
            plan_utterance(plan, in, utt, longest(leff, in, utt, S_max, lane),
                           mixed && (stored_only || !takes_fused_route(*leff_all)), lane);
        return;
    }
    const int id = blockIdx.x - n_plan, part = id % P, us = id / P, utt = us / S_max, s = us - utt * S_max;
    const int from = part * BLK2;
    const AugUttParams &row = table[utt];
    fftpair::fill_tables(sh, t, tw);
    if (row.n_src < 1 || row.n_src > S_max || s >= row.n_src) {
        chain_wait();
        if (LENGTHS == FIND && s == 0 && t < 32)
            plan_utterance(plan, plan_input(plan, row, utt, S_max, t), utt, 1, false, t);
        return;
    }
    chain_wait();
    const int end = LENGTHS == KNOWN ? min(leff[us], L) : L;
    if (part > 0 && from >= end) {
        // (a longer response of the same utterance may be the reason that the products take this partition)
        int most = 0;
        for (int i = 0; i < row.n_src; ++i) most = max(most, leff[utt * S_max + i]);
        if (from >= most) return;
    }
    const float scale = (s == 0 ? 1.f : row.noise_weight[s - 1]) / (4.f * (float)F2);
    const float *h = rir + (int64_t)us * L;
    float4 *out = hspec + ((int64_t)us * P + part) * (NB2 / 2) + t;
    static_assert(4 * CF * (NP2 / 2) == BLK2, "");
    C2 v[NP2];
    int last = 0;
    float4 z[NP2 / 2];
    if ((L & 3) == 0 && (reinterpret_cast<uintptr_t>(rir) & 15) == 0) {
        // rows of whole groups of four
#pragma unroll
        for (int r = 0; r < NP2 / 2; ++r) {
            const int i0 = from + 4 * (t + CF * r);
            z[r] = i0 < end ? *reinterpret_cast<const float4 *>(h + i0) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    } else {
#pragma unroll
        for (int r = 0; r < NP2 / 2; ++r) {
            const int i0 = from + 4 * (t + CF * r);
            z[r] = make_float4(i0 < end ? h[i0] : 0.f, i0 + 1 < end ? h[i0 + 1] : 0.f, i0 + 2 < end ? h[i0 + 2] : 0.f,
                               i0 + 3 < end ? h[i0 + 3] : 0.f);
        }
    }
#pragma unroll
    for (int r = 0; r < NP2 / 2; ++r) {
        const int i0 = from + 4 * (t + CF * r);
        if (LENGTHS == FIND) {
            if (z[r].x != 0.f) last = i0 + 1;
            if (z[r].y != 0.f) last = i0 + 2;
            if (z[r].z != 0.f) last = i0 + 3;
            if (z[r].w != 0.f) last = i0 + 4;
        }
        v[r] = {fftpair::pack(z[r].x, z[r].y), fftpair::pack(z[r].z, z[r].w)};
    }
#pragma unroll
    for (int r = NP2 / 2; r < NP2; ++r) v[r] = {0, 0};
    if (LENGTHS == FIND) {
        last = __reduce_max_sync(0xffffffffu, last);
        if ((t & 31) == 0) red_i[t >> 5] = last;
    }
    __syncthreads();
    // a count of the sources and the length of each in one word
    static_assert(AUG_S_MAX <= 4 && BLK2 < (1 << 14), "");
    unsigned long long sum = 0;
    if (LENGTHS == FIND && t == 0) {
        int m = 0;
#pragma unroll
        for (int i = 0; i < CF / 32; ++i) m = max(m, red_i[i]);
        const unsigned long long mine = (1ull << 56) | ((unsigned long long)m << (14 * s));
        sum = atomicAdd(&arrived[utt], mine) + mine;
    }
    fftpair::forward4096(v, sh, t, tw);
    chain_next();
    fftpair::exchange_mirror(v, t);
    const u64 sc = fftpair::both(scale);
    const float2 u = __ldg(&tw[8192 + fftpair::row_frequency(t)]);
#pragma unroll
    for (int r = 0; r < NS2; ++r) {
        Bins x = r == 0 && fftpair::owns_zero(t) ? edge_forward(v[0], v[NP2 - 1])
                                                 : bins_forward(v[r], v[NP2 - 1 - r], SplitTwiddle(u, r));
        x = {fftpair::mul2(x.pr, sc), fftpair::mul2(x.pi, sc), fftpair::mul2(x.qr, sc), fftpair::mul2(x.qi, sc)};
        store_bins(out + 2 * r * CF, x);
    }
    if (LENGTHS == FIND && t < 32) {
        sum = __shfl_sync(0xffffffffu, sum, 0);
        if ((int)(sum >> 56) == row.n_src) {
            const int len = t < 4 ? (int)(sum >> (14 * t)) & ((1 << 14) - 1) : 0;
            plan_utterance(plan, plan_input(plan, row, utt, S_max, t), utt, __reduce_max_sync(0xffffffffu, len), false, t);
        }
    }
}

// Outputs [from, end) of a block of v that lie behind copy_from, wherever they come back; o = its thread's first group of
// four, the others are 4 CF apart, and all of the block has just been written.  own: the sum of this thread's squares.
// Returns that of the copies'.  Equal ones are counted, not added one by one: in a running sum of all of them a
// constant stretch came out 2e-5 too loud or quiet over 60 s.
// Bound by instructions: 256 utterances of 20 s over stretches of 0.6 of their length 1081 us without copies, 987 with
// squares added up for every block, 974 with those of blocks that come back whole taken from `own`; with stretches
// that are no multiple of 4, 1078, and 1021 with single words at the places of groups, 1000 lane by lane.
__device__ __forceinline__ float repeat_block(float *row, int o, int from, int end, int copy_from, int period, int N, float own) {
    const int first = max(from, copy_from);
    float sum = 0.f;
    if (((period | copy_from) & 3) == 0) {
        const int copies = (N - end) / period;         // of the last output
        if (first == from && (N - 1 - from) / period == copies) {
            // all of the block comes back as often
#pragma unroll 1
            for (; o < end; o += 4 * CF) {
                if (o < from) continue;
                float *p = row + o;
                const float4 y = *reinterpret_cast<const float4 *>(p);
#pragma unroll 1
                for (int k = 0; k < copies; ++k) {
                    p += period;
                    *reinterpret_cast<float4 *>(p) = y;
                }
            }
            return (float)copies * own;
        }
#pragma unroll 1
        for (; o < end; o += 4 * CF) {
            if (o < first) continue;
            const float4 y = *reinterpret_cast<const float4 *>(row + o);
            unsigned m = o + period;
            float whole = 0.f;
#pragma unroll 1
            for (; m + 3 < (unsigned)N; m += period, whole += 1.f) *reinterpret_cast<float4 *>(row + m) = y;
            sum = fmaf(whole, fmaf(y.x, y.x, fmaf(y.y, y.y, fmaf(y.z, y.z, y.w * y.w))), sum);
            if (m < (unsigned)N) {
                // (workspace rows are allocated up to a multiple of 4)
                const float4 z = make_float4(y.x, m + 1 < (unsigned)N ? y.y : 0.f, m + 2 < (unsigned)N ? y.z : 0.f, 0.f);
                *reinterpret_cast<float4 *>(row + m) = z;
                sum = fmaf(z.x, z.x, fmaf(z.y, z.y, fmaf(z.z, z.z, sum)));
            }
        }
    } else {
        // 128 outputs of a warp at a time, lane by lane: stores of whole sectors wherever they go
        const int lane = threadIdx.x & 31;
        __syncwarp();
#pragma unroll 1
        for (o -= 4 * lane; o < end; o += 4 * CF) {
            if (o + 127 < first) continue;
            const bool all = o >= first && o + 128 <= end;
            float *p = row + o + lane;
            float z[4], whole = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int i = o + 32 * c + lane;
                z[c] = i >= first && i < end ? p[32 * c] : 0.f;
            }
            unsigned q = period;
            if (all) {
#pragma unroll 1
                for (; q + 127 < (unsigned)(N - o); q += period, whole += 1.f) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) p[q + 32 * c] = z[c];
                }
            }
            sum = fmaf(whole, fmaf(z[0], z[0], fmaf(z[1], z[1], fmaf(z[2], z[2], z[3] * z[3]))), sum);
#pragma unroll 1
            for (; q < (unsigned)(N - o); q += period) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int i = o + 32 * c + lane;
                    if (i >= first && i < end && q < (unsigned)(N - i)) {
                        p[q + 32 * c] = z[c];
                        sum = fmaf(z[c], z[c], sum);
                    }
                }
            }
        }
    }
    return sum;
}

// KIND  FUSED    a block of one output from its samples (responses of one partition)
//       SPECTRA  the spectra of a block's segments, one per source, stored
//       STORED   a block of one output from stored spectra
// PARK (FUSED): rows may have several noise sources (the context allows three or more
// sources); without it the kernel carries none of the parking code.
//
// Several noise sources are summed in the frequency domain: the products of all but the last
// are parked in a 64 KB global slot of the CTA's own (it stays in L2) and added to the last
// one's before the single inverse transform.  Where the slot is held (park_flags) the sum is
// done in the time domain instead: v is read back and added to for every source after the
// first, one inverse transform each.
//
// FUSED is bound by the issue of instructions, SPECTRA by those and its stores, STORED by the
// latency of the spectra.  FUSED on 256 utterances of 2-20 s: 538 us with scalar transforms, one
// CTA per possible block and three CTAs per multiprocessor (80 registers); 418 with two transforms
// side by side in packed arithmetic, 128 registers, two CTAs and the list of work.
enum Fate { DIRECT = 0, PARK_FIRST = 1, PARK_MORE = 2, PARK_JOIN = 3 };

enum Kind { FUSED, SPECTRA, STORED };

template <Kind KIND, bool PARK>
__global__ void __launch_bounds__(CF, FUSED_MINB)
convolve_kernel(const Plan *plans, const Unit *units, const int *n_units, int unit_cap,
                int *drawn, int S_max, int P, const float4 *hspec, float4 *__restrict__ xspec,
                int nblk_cap, const float2 *__restrict__ tw, float *__restrict__ ys, float *__restrict__ vv,
                int64_t ws_stride, double *__restrict__ energy, float4 *__restrict__ park,
                const int *__restrict__ park_flags) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fftpair::Shared &sh = *reinterpret_cast<fftpair::Shared *>(smem_raw);
    // The first two units of a CTA follow from its number, the others it draws from a counter (units
    // differ: more noise sources, more work; dealt out in turn they left CTAs idle, 567 against
    // 447 us on 256 utterances of 2-20 s).  The unit after next and the next one's plan are
    // fetched while the current one is worked on; a warp may be up to one unit behind, hence three
    // places for each.  The exchange buffer of the unit before may still be read by such a warp (the
    // inverse transform ends with reads of all rows).  FUSED and SPECTRA go on with a forward transform,
    // which first writes the slots its own thread has read last and then waits for all, SPECTRA behind a
    // barrier after its own last reads; STORED goes on with an inverse one, which writes whole rows, and
    // has a barrier behind the one before.
    __shared__ Plan plan_s[3];
    __shared__ Unit unit_s[3];
    __shared__ int3 list_s;                    // sums, those and blocks with copies, all units
    const int t = threadIdx.x, G = gridDim.x;
    fftpair::fill_tables(sh, t, tw);
    chain_wait();
    // (a CTA's first unit, which mostly is one of three, is read beside the counts)
    // SPECTRA goes through the list backwards: the spectra that it writes last are still in L2 when STORED starts
    // (128 x 8 s, four sources: 250 -> 246 us).
    const Unit front = units[blockIdx.x], middle = units[unit_cap + blockIdx.x], back = units[unit_cap - 1 - blockIdx.x];
    const int heavy = n_units[0], early = heavy + n_units[1], count = early + n_units[2];
    if (blockIdx.x >= count) return;
    auto unit_at = [&](int i, int3 n) {
        if (KIND == SPECTRA) i = n.z - 1 - i;
        return units[i < n.x ? i : i < n.y ? unit_cap + (i - n.x) : unit_cap - 1 - (i - n.y)];
    };
    const int3 list = make_int3(heavy, early, count);
    const Unit first = KIND == SPECTRA                          ? unit_at(blockIdx.x, list)
                       : blockIdx.x < heavy                     ? front
                       : heavy == 0 && blockIdx.x < early       ? middle
                       : early == 0                             ? back
                                                                : unit_at(blockIdx.x, list);
    if (t == 32) {
        const int second = blockIdx.x + G;
        list_s = list;
        unit_s[0] = first;
        unit_s[1] = second < count ? unit_at(second, list) : Unit{-1, 0};
    }
    if (t < (int)(sizeof(Plan) / 4))
        reinterpret_cast<int *>(&plan_s[0])[t] = reinterpret_cast<const int *>(plans + first.utt)[t];
    __syncthreads();
    const bool own_slot = KIND == FUSED && PARK && park != nullptr && park_flags[blockIdx.x] == 0;

#pragma unroll 1
    for (int k = 0;;) {
        const Plan &p = plan_s[k];
        const Unit cur = unit_s[k];
        const int k1 = k == 2 ? 0 : k + 1, k2 = k == 0 ? 2 : k - 1;
        const int next_utt = unit_s[k1].utt;
        if (next_utt < 0) chain_next();        // the CTA's last unit
        if (next_utt >= 0 && t < (int)(sizeof(Plan) / 4))
            copy4_async(reinterpret_cast<float *>(&plan_s[k1]) + t,
                        reinterpret_cast<const float *>(plans + next_utt) + t, 4);
        int ticket = 0;
        if (t == 0) ticket = 2 * G + atomicAdd(drawn, 1);
        auto draw = [&]() {                    // (published by the barrier that follows)
            if (t == 0) unit_s[k2] = ticket < list_s.z ? unit_at(ticket, list_s) : Unit{-1, 0};
            copies_done();
        };
        const bool noise = cur.block2 & 1;
        const int b = cur.block2 >> 1;
        // sources of this output: list entries j .. j_last
        int j = noise ? 1 : 0;
        const int j_last = noise ? p.n_noise : 0;
        if (j > j_last || p.n_src == 0) {
            // no (usable) source: the output is defined as silence
            float *dst = (noise ? vv : ys) + (int64_t)cur.utt * ws_stride + (int64_t)b * p.ob;
            const int n_left = min(p.N - b * p.ob, p.ob);
            if (KIND != SPECTRA)
                for (int i = t; i < n_left; i += CF) dst[i] = 0.f;
            draw();
            __syncthreads();
        } else {
            bool added = false;
#pragma unroll 1
            for (;; ++j) {
                C2 v[NP2];
                Fate fate = DIRECT;
                if constexpr (KIND == SPECTRA) {
                    if (j == j_last) draw();
                    else if (t == 0) {
                        // the next source's segment, where it lies in one piece, on its way to L2 meanwhile
                        // (241 -> 238 us)
                        const int nb = (b + 1) * p.ob - F2, nl = p.nlen[j + 1];
                        if (nb >= 0 && nb + F2 <= p.N) {
                            const int m0 = nb % nl;
                            const float *q = p.x[j + 1] + m0;
                            if (m0 + F2 <= nl && (reinterpret_cast<uintptr_t>(q) & 15) == 0)
                                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(q), "n"(4 * F2) : "memory");
                        }
                    }
                    load_segment(v, sh, p.x[j], noise, p.nlen[j], (b + 1) * p.ob - F2, p.N, t);
                    fftpair::forward4096(v, sh, t, tw);
                    float4 *X = xspec + (((int64_t)cur.utt * S_max + p.src[j]) * nblk_cap + b) * (NB2 / 2) + t;
                    const float2 u = __ldg(&tw[8192 + fftpair::row_frequency(t)]);
                    fftpair::exchange_mirror(v, t);
#pragma unroll
                    for (int r = 0; r < NS2; ++r)
                        store_bins(X + 2 * r * CF,
                                   r == 0 && fftpair::owns_zero(t) ? edge_forward(v[0], v[NP2 - 1])
                                                                   : bins_forward(v[r], v[NP2 - 1 - r], SplitTwiddle(u, r)));
                    __syncthreads();           // other warps may still read rows of the buffer the next source fills
                    if (j == j_last) break;
                    continue;
                }
                if constexpr (KIND == STORED) {
                    // All sources of the output and all partitions into one sum.  Bound by the latency of the
                    // spectra (128 KB per product; half of those of the audio come from memory): the next
                    // product's are brought into L2 while one is worked on, and each slot's are
                    // requested one slot ahead (319 -> 248 us on 128 x 8 s).
                    Bins acc[NS2], xa, ha;
#pragma unroll
                    for (int r = 0; r < NS2; ++r) acc[r] = {0, 0, 0, 0};
                    const int parts = min(p.parts, b + 1);
#pragma unroll 1
                    for (; j <= j_last; ++j) {
                        const int64_t row = (int64_t)cur.utt * S_max + p.src[j];
                        const float4 *H = hspec + row * P * (NB2 / 2) + t;
                        const float4 *X = xspec + (row * nblk_cap + b) * (NB2 / 2) + t;
                        xa = load_parked(X);
                        ha = load_bins(H);
#pragma unroll 1
                        for (int q = 0; q < parts; ++q) {
                            const bool more = q + 1 < parts;
                            if (t == 0 && (more || j < j_last)) {
                                const int64_t row_n = (int64_t)cur.utt * S_max + p.src[min(j + 1, j_last)];
                                prefetch_spectrum(more ? H + NB2 / 2 : hspec + row_n * P * (NB2 / 2));
                                prefetch_spectrum(more ? X - NB2 / 2 : xspec + (row_n * nblk_cap + b) * (NB2 / 2));
                            }
#pragma unroll
                            for (int r = 0; r < NS2; ++r) {
                                using namespace fftpair;
                                Bins x = xa;
                                const Bins h = ha;
                                if (r + 1 < NS2 || more) {
                                    xa = load_parked(r + 1 < NS2 ? X + 2 * (r + 1) * CF : X - NB2 / 2);
                                    ha = load_bins(r + 1 < NS2 ? H + 2 * (r + 1) * CF : H + NB2 / 2);
                                }
                                if (r == 0 && owns_zero(t)) {
                                    edge_multiply(x, h);
                                    acc[0] = {add2(acc[0].pr, x.pr), add2(acc[0].pi, x.pi), add2(acc[0].qr, x.qr),
                                              add2(acc[0].qi, x.qi)};
                                } else {
                                    acc[r].pr = sub2(fma2(x.pr, h.pr, acc[r].pr), mul2(x.pi, h.pi));
                                    acc[r].pi = fma2(x.pi, h.pr, fma2(x.pr, h.pi, acc[r].pi));
                                    acc[r].qr = sub2(fma2(x.qr, h.qr, acc[r].qr), mul2(x.qi, h.qi));
                                    acc[r].qi = fma2(x.qi, h.qr, fma2(x.qr, h.qi, acc[r].qi));
                                }
                            }
                            H += NB2 / 2;
                            X -= NB2 / 2;
                        }
                    }
                    j = j_last;
                    const float2 u = __ldg(&tw[8192 + fftpair::row_frequency(t)]);
#pragma unroll
                    for (int r = 0; r < NS2; ++r) {
                        if (r == 0 && fftpair::owns_zero(t)) edge_inverse(acc[0], v[0], v[NP2 - 1]);
                        else bins_inverse(acc[r], SplitTwiddle(u, r), v[r], v[NP2 - 1 - r]);
                    }
                }
                if constexpr (KIND == FUSED) {
                    if (PARK && own_slot && j_last > 1)
                        fate = j == j_last ? PARK_JOIN : j > 1 ? PARK_MORE : PARK_FIRST;
                    load_segment(v, sh, p.x[j], noise, p.nlen[j], (b + 1) * p.ob - F2, p.N, t);
                    // the response's bins are brought into L2 meanwhile (they may have been pushed out by the
                    // audio), and the first two slots' requested before the exchange
                    const float4 *H = hspec + ((int64_t)cur.utt * S_max + p.src[j]) * P * (NB2 / 2) + t;
                    if (t == 0) prefetch_spectrum(H);
                    fftpair::forward4096(v, sh, t, tw);
                    Bins h = load_bins(H), h1 = load_bins(H + 2 * CF);
                    const float2 u = __ldg(&tw[8192 + fftpair::row_frequency(t)]);
                    fftpair::exchange_mirror(v, t);
#pragma unroll
                    for (int r = 0; r < NS2; ++r) {
                        const Bins hc = h;
                        h = h1;
                        if (r + 2 < NS2) h1 = load_bins(H + 2 * (r + 2) * CF);
                        const bool edge = r == 0 && fftpair::owns_zero(t);
                        const SplitTwiddle w(u, r);
                        Bins y;
                        if (edge) {
                            y = edge_forward(v[0], v[NP2 - 1]);
                            edge_multiply(y, hc);
                        } else {
                            y = bins_forward(v[r], v[NP2 - 1 - r], w);
                            multiply(y.pr, y.pi, hc.pr, hc.pi);
                            multiply(y.qr, y.qi, hc.qr, hc.qi);
                        }
                        if (PARK && fate != DIRECT) {
                            // this thread's parked products, two words per slot: no other thread reads them
                            float4 *pk = park + (int64_t)blockIdx.x * (2 * NS2 * CF) + 2 * r * CF + t;
                            if (fate != PARK_FIRST) {
                                const Bins z = load_parked(pk);
                                y = {fftpair::add2(y.pr, z.pr), fftpair::add2(y.pi, z.pi), fftpair::add2(y.qr, z.qr),
                                     fftpair::add2(y.qi, z.qi)};
                            }
                            if (fate != PARK_JOIN) store_bins(pk, y);
                        }
                        if (edge) edge_inverse(y, v[0], v[NP2 - 1]);
                        else bins_inverse(y, w, v[r], v[NP2 - 1 - r]);
                    }
                    if (PARK && (fate == PARK_FIRST || fate == PARK_MORE)) {
                        __syncthreads();       // other warps may still read rows of the buffer the next source fills
                        continue;
                    }
                }
                fftpair::exchange_back(v, t);
                if (j == j_last) draw();
                fftpair::inverse4096(v, sh, t, tw);
                // (here, where the warps are close together, 128 x 8 s with 24000 taps take what they took
                // without it, 863 us; between the products and the inverse transform it cost 5)
                if constexpr (KIND == STORED) __syncthreads();

                // The last `ob` outputs of the segment are this block: samples 4m .. 4m+3 of the
                // segment are point m = t + CF r, real and imaginary parts swapped.
                const int ob = p.ob, n_left = min(p.N - b * ob, ob);
                float *dst = (noise ? vv : ys) + (int64_t)cur.utt * ws_stride + (int64_t)b * ob;
                u64 e2 = 0;
                const int o0 = 4 * t - (F2 - ob);         // first of this thread's outputs, 4 CF apart
                if (n_left == ob && !(PARK && added)) {
                    // a whole block (most are)
#pragma unroll
                    for (int r = 0; r < NP2; ++r) {
                        if (o0 + 4 * CF * r >= 0) {
                            const float2 lo = fftpair::unpack(v[r].im), hi = fftpair::unpack(v[r].re);
                            *reinterpret_cast<float4 *>(dst + o0 + 4 * CF * r) = make_float4(lo.x, lo.y, hi.x, hi.y);
                            e2 = fftpair::fma2(v[r].re, v[r].re, fftpair::fma2(v[r].im, v[r].im, e2));
                        }
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < NP2; ++r) {
                        const int o = o0 + 4 * CF * r;
                        if (o >= 0 && o < n_left) {
                            const float2 lo = fftpair::unpack(v[r].im), hi = fftpair::unpack(v[r].re);
                            // (workspace rows are allocated up to a multiple of 4)
                            float4 y = make_float4(lo.x, o + 1 < n_left ? lo.y : 0.f, o + 2 < n_left ? hi.x : 0.f,
                                                   o + 3 < n_left ? hi.y : 0.f);
                            float4 *q = reinterpret_cast<float4 *>(dst + o);
                            if (PARK && added) {
                                const float4 z = *q;
                                y = make_float4(y.x + z.x, y.y + z.y, y.z + z.z, y.w + z.w);
                            }
                            *q = y;
                            const u64 a = fftpair::pack(y.x, y.y), c = fftpair::pack(y.z, y.w);
                            e2 = fftpair::fma2(a, a, fftpair::fma2(c, c, e2));
                        }
                    }
                }
                added = true;
                if (j == j_last) {
                    const float2 e = fftpair::unpack(e2);
                    float sum = e.x + e.y;
                    if (KIND == FUSED && noise && p.period > 0 && (b + 1) * ob > p.copy_from)
                        sum += repeat_block(dst - (int64_t)b * ob, b * ob + o0, b * ob, (b + 1) * ob, p.copy_from, p.period,
                                            p.N, sum);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                    if ((t & 31) == 0) atomicAdd(&energy[2 * cur.utt + (noise ? 1 : 0)], (double)sum);
                    break;
                }
                if (PARK) __syncthreads();
            }
        }
        if (next_utt < 0) break;
        k = k1;
    }
}

constexpr size_t FFT2_SMEM = sizeof(fftpair::Shared);

}  // namespace

static bool stored_route(const AugCtx *ctx) { return ctx->route == aug::ROUTE_STORED; }

// Most units of work that a batch can have, with blocks of ob outputs.
static int64_t most_units(int max_len, int B, int ob) { return 2 * (int64_t)B * (((int64_t)max_len + ob - 1) / ob); }
// blocks of the fused kernel are shortest where a response fills min(rir_taps, 8192) taps
static int shortest_block(const AugCtx *ctx) { return (F2 - std::min(ctx->cfg.rir_taps, BLK2) + 1) & ~3; }

static PlanArgs plan_args(const AugCtx *ctx, const ConvInput &in) {
    // Copies lengthen the units that make them, which does not pay before other units wait for a place: one utterance
    // of 60 s over a stretch of 1 s 46 us computed, 89 copied (of 16001 samples 48 and 234), eight of 2 s 31 and 33.
    // What counts is the largest batch that the context is for, so that an utterance's numbers do not depend on those
    // it comes with, nor on the chunks of the host entry point (one of 20 s over 0.25 to 1 s in a context for hundreds:
    // 40 us computed, 46 copied).  Blocks are up to twice as long as the shortest, hence two rounds.
    const int repeats = most_units(ctx->cfg.max_samples, ctx->cfg.max_batch, shortest_block(ctx)) >
                        2 * (int64_t)FUSED_MINB * ctx->sm_count;
    return {in.speech, in.stride, in.lengths, in.bank, in.bank_len, in.max_len, ctx->status,
            reinterpret_cast<Plan *>(ctx->plans), reinterpret_cast<Unit *>(ctx->units), ctx->unit_cap, ctx->counters,
            repeats};
}

template <Lengths LENGTHS>
static int launch_spectra(AugCtx *ctx, const float *rir, const ConvInput &in, const AugUttParams *table, int B,
                          int n_plan) {
    const AugConfig &c = ctx->cfg;
    if (smem_opt_in<rir_spectra2_kernel<LENGTHS>>(ctx->device) != AUG_OK) return AUG_ECUDA;
    if (launch_chained(rir_spectra2_kernel<LENGTHS>, dim3(n_plan + ctx->n_part * c.max_sources * B), CF, FFT2_SMEM,
                       ctx->stream, rir, table, B, c.max_sources, c.rir_taps, ctx->n_part, ctx->tw,
                       reinterpret_cast<float4 *>(ctx->hspec), ctx->leff, ctx->arrived, plan_args(ctx, in), n_plan,
                       ctx->counters + aug::LEFF_ALL, stored_route(ctx) ? 1 : 0, ctx->stored_only) != AUG_OK)
        return AUG_ECUDA;
    ctx->launches++;
    return AUG_OK;
}

int launch_rir_spectra(AugCtx *ctx, const float *rir, const ConvInput &in, const AugUttParams *table, int B,
                       bool measured) {
    const AugConfig &c = ctx->cfg;
    const bool mixed = stored_route(ctx);
    // long-response context: the last batch size seen decides whether the fused kernels are launched at all
    ctx->stored_only = mixed && ctx->leff_seen && *ctx->leff_seen > BLK2;
    if (measured) return launch_spectra<KNOWN>(ctx, rir, in, table, B, (B + CF / 32 - 1) / (CF / 32));
    AUG_CUDA_OK(cudaMemsetAsync(ctx->energy, 0, reinterpret_cast<char *>(ctx->counters + aug::N_COUNTERS) -
                                                    reinterpret_cast<char *>(ctx->energy), ctx->stream));
    if (!mixed) return launch_spectra<FIND>(ctx, rir, in, table, B, 0);
    if (launch_chained(rir_length_kernel, dim3(c.max_sources, B), CT, 0, ctx->stream, rir, table, c.max_sources,
                       c.rir_taps, ctx->leff, ctx->counters + aug::LEFF_ALL) != AUG_OK)
        return AUG_ECUDA;
    ctx->launches++;
    return launch_spectra<KNOWN>(ctx, rir, in, table, B, 0);
}

template <Kind KIND, bool PARK>
static int launch_convolve(AugCtx *ctx, int grid) {
    const AugConfig &c = ctx->cfg;
    int *counters = ctx->counters;
    if (smem_opt_in<convolve_kernel<KIND, PARK>>(ctx->device) != AUG_OK) return AUG_ECUDA;
    const int list = KIND == FUSED ? aug::LIST_FUSED : aug::LIST_STORED;
    const int drawn = KIND == FUSED ? aug::DRAWN_FUSED : KIND == SPECTRA ? aug::DRAWN_SPECTRA : aug::DRAWN_STORED;
    if (launch_chained(convolve_kernel<KIND, PARK>, dim3(grid), CF, FFT2_SMEM, ctx->stream,
                       reinterpret_cast<const Plan *>(ctx->plans), reinterpret_cast<const Unit *>(ctx->units),
                       counters + list, ctx->unit_cap, counters + drawn, c.max_sources, ctx->n_part,
                       reinterpret_cast<const float4 *>(ctx->hspec), reinterpret_cast<float4 *>(ctx->xspec),
                       ctx->nblk_cap, ctx->tw, ctx->ys, ctx->vv, ctx->ws_stride, ctx->energy, ctx->park,
                       ctx->park_flags) != AUG_OK)
        return AUG_ECUDA;
    ctx->launches++;
    return AUG_OK;
}
// As many CTAs as fit (less the room to be left for kernels of other streams), but not more than there
// can be units of work.
static int convolve_grid(const AugCtx *ctx, const ConvInput &in, int B, int ob) {
    const int fit = std::min(FUSED_MINB * ctx->sm_count - in.room, aug::PARK_SLOTS);
    return (int)std::min<int64_t>(most_units(in.max_len, B, ob), fit);
}

int launch_convolve_prepare(AugCtx *ctx, const ConvInput &in, const AugUttParams *table, int B, bool measured) {
    const AugConfig &c = ctx->cfg;
    if (in.max_len <= 0 || !stored_route(ctx)) return AUG_OK;
    if (!measured) {
        if (launch_chained(plan_kernel, dim3((B + 7) / 8), 256, 0, ctx->stream, plan_args(ctx, in), table, B,
                           c.max_sources, ctx->leff, ctx->counters + aug::LEFF_ALL, ctx->stored_only) != AUG_OK)
            return AUG_ECUDA;
        ctx->launches++;
    }
    return launch_convolve<SPECTRA, false>(ctx, convolve_grid(ctx, in, B, BLK2));
}

int launch_convolve_finish(AugCtx *ctx, const ConvInput &in, const AugUttParams *table, int B) {
    if (in.max_len <= 0) return AUG_OK;
    int rc = AUG_OK;
    if (!ctx->stored_only) {
        const int grid = convolve_grid(ctx, in, B, shortest_block(ctx));
        rc = ctx->park ? launch_convolve<FUSED, true>(ctx, grid) : launch_convolve<FUSED, false>(ctx, grid);
        if (rc != AUG_OK) return rc;
    }
    if (stored_route(ctx)) {
        if ((rc = launch_convolve<STORED, false>(ctx, convolve_grid(ctx, in, B, BLK2))) != AUG_OK) return rc;
        // for the next call's choice (not waited for)
        if (ctx->leff_seen)
            AUG_CUDA_OK(cudaMemcpyAsync(ctx->leff_seen, ctx->counters + aug::LEFF_ALL, sizeof(int), cudaMemcpyDeviceToHost,
                                        ctx->stream));
    }
    return AUG_OK;
}

int launch_snr_gain(AugCtx *ctx, const AugUttParams *table, int B) {
    if (launch_chained(snr_gain_kernel, dim3((B + 255) / 256), 256, 0, ctx->stream, ctx->energy, table, B, ctx->gain) !=
        AUG_OK)
        return AUG_ECUDA;
    ctx->launches++;
    return AUG_OK;
}

int launch_mix(AugCtx *ctx, const int *lengths, const AugUttParams *table, int B, int max_len, bool ready,
               float *wave_out, int64_t out_stride) {
    if (max_len <= 0) return AUG_OK;
    dim3 grid((max_len + MIX_GROUPS * 1024 - 1) / (MIX_GROUPS * 1024), B);
    const GainSource gain = {ready ? ctx->gain : nullptr, ctx->energy, table};
    if (launch_chained(ready ? mix_kernel<true> : mix_kernel<false>, grid, 256, 0, ctx->stream, ctx->ys, ctx->vv,
                       ctx->ws_stride, gain, lengths, wave_out, out_stride, max_len) != AUG_OK)
        return AUG_ECUDA;
    ctx->launches++;
    return AUG_OK;
}
