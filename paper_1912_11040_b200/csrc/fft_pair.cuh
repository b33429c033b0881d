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
// half: 1).
__device__ __forceinline__ void fft512(C2 *v, u64 *buf, float4 c, int l) {
    dft16(v);
    twiddle16(v, make_float2(c.x, c.y));
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

}  // namespace fftpair
