// Two complex transforms side by side in packed fp32 arithmetic.
//
// add / sub / mul / fma.rn.f32x2 do two fp32 operations per lane and instruction.  They run at
// the arithmetic rate of the scalar forms (measured: 1.96 packed against 3.8 scalar warp
// instructions per clock and multiprocessor), so they do not raise the fp32 peak; they
// halve the issue slots, and a pair of equal transforms needs no shuffling of operands to
// use them: a number here is the real (or imaginary) part of the same point of transform A
// and of transform B.
#pragma once
#include <cuda_runtime.h>

namespace fftpair {

// Twiddle table, TW_N entries: for every power of two M <= TW_N the block
// [M/2, M) holds exp(-2 pi i k / M), k < M/2, so that the factors one pass or one
// real-FFT split needs are contiguous in k (coalesced loads).
constexpr int TW_N = 16384;
__host__ __device__ constexpr int tw_index(int M, int k) { return M / 2 + k; }

typedef unsigned long long u64;

__device__ __forceinline__ u64 pack(float lo, float hi) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack(u64 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ u64 both(float x) { return pack(x, x); }
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ u64 sub2(u64 a, u64 b) {
    u64 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// The same point of both transforms.
struct C2 {
    u64 re, im;
};
__device__ __forceinline__ C2 add(C2 a, C2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ C2 sub(C2 a, C2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
// One factor for both transforms.
struct W2 {
    u64 x, y;
};
__device__ __forceinline__ W2 both(float2 w) { return {both(w.x), both(w.y)}; }
__device__ __forceinline__ C2 times(C2 v, W2 w) {
    return {sub2(mul2(w.x, v.re), mul2(w.y, v.im)), fma2(w.y, v.re, mul2(w.x, v.im))};
}
__device__ __forceinline__ W2 times(W2 a, W2 b) {
    return {sub2(mul2(a.x, b.x), mul2(a.y, b.y)), fma2(a.x, b.y, mul2(a.y, b.x))};
}

// In-register DFTs (e^{-i...}), natural order in and out; the factors between the radix-2
// steps are folded into fused multiply-adds (c (1 + i t) with t the tangent).
__device__ __forceinline__ void dft4(C2 &a, C2 &b, C2 &c, C2 &d) {
    const C2 t0 = add(a, c), t1 = sub(a, c), t2 = add(b, d), t3 = sub(b, d);
    a = add(t0, t2);
    c = sub(t0, t2);
    b = {add2(t1.re, t3.im), sub2(t1.im, t3.re)};
    d = {sub2(t1.re, t3.im), add2(t1.im, t3.re)};
}
// (e + c (x, y), e - c (x, y))
__device__ __forceinline__ void join(C2 e, u64 c, u64 nc, u64 x, u64 y, C2 &p, C2 &m) {
    p = {fma2(c, x, e.re), fma2(c, y, e.im)};
    m = {fma2(nc, x, e.re), fma2(nc, y, e.im)};
}
// (e + c (x, -y), e - c (x, -y))
__device__ __forceinline__ void join_n(C2 e, u64 c, u64 nc, u64 x, u64 y, C2 &p, C2 &m) {
    p = {fma2(c, x, e.re), fma2(nc, y, e.im)};
    m = {fma2(nc, x, e.re), fma2(c, y, e.im)};
}
__device__ __forceinline__ void dft8(C2 *v) {
    const u64 h = both(0.70710678118654752440f), nh = both(-0.70710678118654752440f);
    C2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4(e0, e1, e2, e3);
    dft4(o0, o1, o2, o3);
    v[0] = add(e0, o0);
    v[4] = sub(e0, o0);
    join(e1, h, nh, add2(o1.re, o1.im), sub2(o1.im, o1.re), v[1], v[5]);
    v[2] = {add2(e2.re, o2.im), sub2(e2.im, o2.re)};
    v[6] = {sub2(e2.re, o2.im), add2(e2.im, o2.re)};
    join_n(e3, h, nh, sub2(o3.im, o3.re), add2(o3.re, o3.im), v[3], v[7]);
}
__device__ __forceinline__ void dft16(C2 *v) {
    C2 e[8], o[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        e[k] = v[2 * k];
        o[k] = v[2 * k + 1];
    }
    dft8(e);
    dft8(o);
    const u64 h = both(0.70710678118654752440f), nh = both(-0.70710678118654752440f);
    const u64 c = both(0.92387953251128675613f), nc = both(-0.92387953251128675613f);   // cos(pi/8)
    const u64 t = both(0.41421356237309504880f), nt = both(-0.41421356237309504880f);   // tan(pi/8)
    v[0] = add(e[0], o[0]);
    v[8] = sub(e[0], o[0]);
    join(e[1], c, nc, fma2(t, o[1].im, o[1].re), fma2(nt, o[1].re, o[1].im), v[1], v[9]);
    join(e[2], h, nh, add2(o[2].re, o[2].im), sub2(o[2].im, o[2].re), v[2], v[10]);
    join_n(e[3], c, nc, fma2(t, o[3].re, o[3].im), fma2(nt, o[3].im, o[3].re), v[3], v[11]);
    v[4] = {add2(e[4].re, o[4].im), sub2(e[4].im, o[4].re)};
    v[12] = {sub2(e[4].re, o[4].im), add2(e[4].im, o[4].re)};
    join_n(e[5], c, nc, fma2(nt, o[5].re, o[5].im), fma2(t, o[5].im, o[5].re), v[5], v[13]);
    join_n(e[6], h, nh, sub2(o[6].im, o[6].re), add2(o[6].re, o[6].im), v[6], v[14]);
    join(e[7], nc, c, fma2(nt, o[7].im, o[7].re), fma2(t, o[7].re, o[7].im), v[7], v[15]);
}

// v[r] *= w^r.  The powers are built by squaring and one more product each, so that none is
// more than four roundings away from w; in packed form too, as a scalar product and the moves
// that double it take more issue slots.
__device__ __forceinline__ void twiddle16(C2 *v, float2 w) {
    const W2 w1 = both(w), w2 = times(w1, w1), w3 = times(w2, w1), w4 = times(w2, w2);
    v[1] = times(v[1], w1);
    v[2] = times(v[2], w2);
    v[3] = times(v[3], w3);
    W2 q = w4;
#pragma unroll
    for (int r = 4; r < 16; r += 4) {
        v[r] = times(v[r], q);
        v[r + 1] = times(v[r + 1], times(q, w1));
        v[r + 2] = times(v[r + 2], times(q, w2));
        v[r + 3] = times(v[r + 3], times(q, w3));
        q = r == 4 ? times(w4, w4) : times(q, w4);
    }
}

// v[r] *= w[(r - 1) STEP], factors doubled (x, x, y, y)
template <int STEP>
__device__ __forceinline__ void twiddle_table(C2 *v, const float4 *w) {
#pragma unroll
    for (int r = 1; r < 16; ++r) {
        const ulonglong2 z = *reinterpret_cast<const ulonglong2 *>(w + (r - 1) * STEP);
        v[r] = times(v[r], W2{z.x, z.y});
    }
}

__device__ __forceinline__ u64 shfl(u64 v, int lane) {
    const float2 z = unpack(v);
    return pack(__shfl_sync(0xffffffffu, z.x, lane), __shfl_sync(0xffffffffu, z.y, lane));
}

// A pair of 512-point transforms by one warp.  Lane l brings the points l + 32 r and ends up
// with the frequencies l + 32 r:  radix 16 over r in registers, the 32 lanes' radix 2 by
// shuffles, the 16 x 16 exchange within each half of the warp through `buf` (XBUF words of 8
// bytes, real parts first, then imaginary parts; rows of 17 keep both patterns free of bank
// conflicts), radix 16 in registers.  One exchange through shared memory where radix-8
// passes need two.
constexpr int XBUF = 32 * 17;
// c: exp(-2 pi i l / 512) and, for the upper half of the warp, exp(-2 pi i (l - 16) / 32) (lower
// half: 1).  TABLE: the factors exp(-2 pi i l r / 512) of the first step come from w[32 (r - 1)],
// each rounded once; built from powers of the first one they double the error of the transform
// (root mean square 2.5e-7 of the spectrum against 1.1e-7).
template <bool TABLE>
__device__ __forceinline__ void fft512(C2 *v, u64 *buf, float4 c, int l, const float4 *w = nullptr) {
    dft16(v);
    if constexpr (TABLE) twiddle_table<32>(v, w);
    else twiddle16(v, make_float2(c.x, c.y));
    const u64 sign = both(l < 16 ? 1.f : -1.f);
    const W2 wh = both(make_float2(c.z, c.w));
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const C2 o = {shfl(v[r].re, l ^ 16), shfl(v[r].im, l ^ 16)};
        v[r] = times(C2{fma2(sign, v[r].re, o.re), fma2(sign, v[r].im, o.im)}, wh);
    }
    u64 *row = buf + 17 * l;
    const u64 *col = buf + 17 * (l & 16) + (l & 15);
#pragma unroll
    for (int r = 0; r < 16; ++r) row[r] = v[r].re;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r].re = col[17 * r];
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 16; ++r) row[r] = v[r].im;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r].im = col[17 * r];
    __syncwarp();
    dft16(v);
}

// A pair of 4096-point transforms by a CTA of 256 threads, 16 points each, in place in shared
// memory: three radix-16 passes.  Digits of an index: slot = 256 a + 16 b + c.
//   forward  pass 1: thread t = 16 b + c transforms the slots 256 r + t over r
//            pass 2: thread (a, c)       the slots 256 a + 16 r + c
//            pass 3: thread (a, b)       the slots 256 a + 16 b + r; its outputs, which stay in
//                    registers, are the frequencies j + 256 r, j = a + 16 b
//   inverse  the same three passes in the opposite order, from frequencies in the registers
//            of thread (a, b) to samples t + 256 r in the registers of thread t.
// Every pass writes the slots it has read, so nothing is overwritten that another thread
// still wants, and as passes 2 and 3 of the forward and 1 and 2 of the inverse direction
// with the same digit a are done by the same warp (two values of a per warp), only the
// boundary between passes 1 and 2 (inverse: 2 and 3) needs a barrier of the whole CTA.
// Real and imaginary parts lie in separate planes of 8-byte words: a 16-byte word would want
// both pairs of registers side by side, which costs moves.  Rows of 16 words are padded by
// one, which keeps all three access patterns free of bank conflicts.
constexpr int THREADS = 256;
constexpr int PLANE = 4096 + 256;
__host__ __device__ constexpr int slot(int i) { return i + (i >> 4); }

// Frequency j = a + 16 b of thread t, whose row of 16 slots is 256 a + 16 b and whose
// frequencies are j + 256 r.  Warp w works on the digits a = w and 16 - w (w = 0: 8 and 0).
// Lane and partner (lane ^ 16) own frequencies that mirror each other:
// 4096 - (j + 256 r) = j' + 256 (15 - r).  j = 128 mirrors itself, and so does j = 0 but with
// 256 (16 - r); these two threads are their own partners.
__host__ __device__ constexpr int row_frequency(int t) {
    const int w = t >> 5, l = t & 31, q = l & 7;
    if (w != 0) return l < 16 ? w + 16 * l : 16 - w + 16 * (31 - l);
    // warp 0: lanes 0-7 and 16-23 a = 8, b and 15 - b; lanes 8-15 and 24-31 a = 0, 16 - b and b
    if (l & 8) return 16 * (l >= 16 ? q : q ? 16 - q : 8);
    return 8 + 16 * (l < 16 ? q : 15 - q);
}
__device__ __forceinline__ bool owns_zero(int t) { return t == 24; }               // j = 0
__device__ __forceinline__ int partner_of(int t) { return (t & ~16) == 8 ? t : (t & 31) ^ 16; }
// Digit a of a thread in pass 2: one per half of the warp.
__device__ __forceinline__ int col_digit(int t) {
    const int w = t >> 5;
    return (t & 16) ? (w ? 16 - w : 0) : (w ? w : 8);
}

struct Shared {
    u64 re[PLANE], im[PLANE];
    float4 w256[15][16];            // exp(-2 pi i k r / 256), doubled (x, x, y, y)
};
// tw: exp(-2 pi i k / M) at M / 2 + k.  The caller synchronises.
__device__ __forceinline__ void fill_tables(Shared &sh, int t, const float2 *__restrict__ tw) {
    if (t < 15 * 16) {
        const int k = ((t >> 4) + 1) * (t & 15);
        float2 w = __ldg(&tw[128 + (k & 127)]);
        if (k & 128) w = make_float2(-w.x, -w.y);
        (&sh.w256[0][0])[t] = make_float4(w.x, w.x, w.y, w.y);
    }
}
template <int STEP>
__device__ __forceinline__ void load16(C2 *v, const Shared &sh, int at) {
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r].re = sh.re[at + STEP * r];
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r].im = sh.im[at + STEP * r];
}
template <int STEP>
__device__ __forceinline__ void store16(const C2 *v, Shared &sh, int at) {
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        sh.re[at + STEP * r] = v[r].re;
        sh.im[at + STEP * r] = v[r].im;
    }
}
__device__ __forceinline__ int row_slot(int t) {
    const int j = row_frequency(t);
    return slot(256 * (j & 15) + (j & ~15));
}
__device__ __forceinline__ int col_slot(int t) { return slot(256 * col_digit(t)) + (t & 15); }

// Samples t + 256 r in v -> frequencies j + 256 r in v.  The slots t + 256 r must be free for
// this thread.
__device__ __forceinline__ void forward4096(C2 *v, Shared &sh, int t, const float2 *__restrict__ tw) {
    const float2 w1 = __ldg(&tw[2048 + t]);
    dft16(v);
    twiddle16(v, w1);
    store16<slot(256)>(v, sh, slot(t));
    __syncthreads();
    load16<slot(16)>(v, sh, col_slot(t));
    dft16(v);
    twiddle_table<16>(v, &sh.w256[0][t & 15]);
    store16<slot(16)>(v, sh, col_slot(t));
    __syncwarp();
    load16<1>(v, sh, row_slot(t));
    dft16(v);
}
// Frequencies j + 256 r in v, real and imaginary parts swapped -> 4096 times the samples
// t + 256 r, swapped too.  The row of slots that holds the thread's frequencies must be free: where
// the thread has not just read it itself (forward4096), all threads must have passed a barrier since
// the buffer was last read.
__device__ __forceinline__ void inverse4096(C2 *v, Shared &sh, int t, const float2 *__restrict__ tw) {
    const float2 w1 = __ldg(&tw[2048 + row_frequency(t)]);
    dft16(v);
    twiddle16(v, w1);
    store16<1>(v, sh, row_slot(t));
    __syncwarp();
    load16<slot(16)>(v, sh, col_slot(t));
    dft16(v);
    twiddle_table<16>(v, &sh.w256[0][col_digit(t)]);
    store16<slot(16)>(v, sh, col_slot(t));
    __syncthreads();
    load16<slot(256)>(v, sh, slot(t));
    dft16(v);
}
// Give the partner frequencies v[8..15] and take its own: v[15 - r] becomes frequency
// 4096 - (j + 256 r) for r < 8 (thread j = 0: for 0 < r < 8, and v[15] becomes frequency 2048).
__device__ __forceinline__ void exchange_mirror(C2 *v, int t) {
    const int partner = partner_of(t);
    if (owns_zero(t)) {
        const C2 x = v[8];
#pragma unroll
        for (int r = 8; r < 15; ++r) v[r] = v[r + 1];
        v[15] = x;
    }
    __syncwarp();
#pragma unroll
    for (int r = 8; r < 16; ++r) v[r] = {shfl(v[r].re, partner), shfl(v[r].im, partner)};
}
// The way back.
__device__ __forceinline__ void exchange_back(C2 *v, int t) {
    const int partner = partner_of(t);
#pragma unroll
    for (int r = 8; r < 16; ++r) v[r] = {shfl(v[r].re, partner), shfl(v[r].im, partner)};
    if (owns_zero(t)) {
        const C2 x = v[15];
#pragma unroll
        for (int r = 15; r > 8; --r) v[r] = v[r - 1];
        v[8] = x;
    }
    __syncwarp();
}

}  // namespace fftpair
