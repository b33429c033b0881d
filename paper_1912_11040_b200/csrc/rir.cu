// Step 1: room impulse responses by the image-source method.
//
// One CTA builds one impulse response (one utterance, one source) in shared
// memory.  Every warp works through batches of 32 images in two phases:
//
//   A  one image per lane: lattice point, distance and delay in fp64 (the delay
//      reaches 2.4e4 samples, where one fp32 ulp is 2e-3 samples), split into
//      an integer n0 and a fraction phi; the five numbers the taps need are
//      written, compacted over the images that contribute, to a slot of a small
//      shared-memory ring owned by the warp.
//   B  four images at a time, their 2 W_h taps over the lanes: lane l owns taps l and l + 32
//      of all four, and of the 16 taps that are left (W_h = 40) the lower half-warp does those
//      of the first two images and the upper half those of the others.  Everything that
//      depends only on the tap sits in registers, and the images' numbers arrive as pairs, the
//      operands of packed (f32x2) arithmetic, by broadcast loads.  With tau = n0 + phi, 0 <= phi < 1,
//      sin(pi (n - tau)) = -(-1)^(n - n0) sin(pi phi), so tap j is As(phi) times
//      (1 + cos(pi (j - phi) / W_h)) / (j - phi).  n0 is rounded down so that the window always
//      covers the same taps -W_h + 1 .. W_h and none has to be masked.  The 32 taps around the
//      centre take a reciprocal and the angle-sum identity of the Hann factor (three fused
//      multiply-adds); W_h >= 40 leaves the others at least eight samples away from the image, where that
//      function of phi is a polynomial of degree four (the first 32 taps) or three (the last 16) to 3e-9 of
//      the image's amplitude, less than the rounding of the reciprocal form (5e-9).  The last multiply-add
//      adds 1.5 2^23, which leaves the fixed-point value in the low bits, and one shared-memory reduction
//      follows.
//
//      Phase A orders the images of a batch: loud ones (their taps need more than 22 bits) first,
//      then the others whose window lies inside the response, then those at its edges, which are
//      done one by one with tests.  No test is left in the loops over the first two.
//
// Bound by instruction issue (26 warp instructions an image, 68 % of the slots) and shared memory (67 % of its
// cycles).  128 x 4 responses of 24000 taps, order 20: 393 us one image at a time in scalar arithmetic, 312
// with two at a time in packed arithmetic, 251 with four at a time and all taps by reciprocals (30
// instructions an image), 228 with polynomials away from the centre, the lattice without searches, the sines as
// series and the tap constants from a table; 512 x up to 4 of 8192 taps, order 12: 162 and 147; 4096 x 2 of
// 4096 taps: 281 and 257.
//
// The response is accumulated in 32-bit fixed point: a shared-memory fp32 atomic
// add is a compare-and-swap loop on this hardware, an integer one is a single
// instruction.  The scale is a power of two chosen per response from the direct
// path, the largest single contribution (A0 = 1/d0): full scale is 64 A0, one
// step 3e-8 A0 (coarser steps show in narrow mel bands that fall into a notch of
// the room's transfer function).  Integer sums are exact, so only the final value
// of a sample has to fit: with fully reflecting walls and order 32 the largest
// sample is 2-3 A0 in rooms of a few metres and 14 A0 in a 30 cm box; a sample
// beyond 64 A0 (rooms of a few centimetres) would wrap.
//
// The lattice points with |kx|+|ky|+|kz| <= order are enumerated compactly in closed
// form (slab kx, then inside the diamond of (ky, kz)), so every lane of a warp carries a real image.
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "fft_pair.cuh"
#include "image_delay.cuh"

namespace {

constexpr int AX = 2 * aug::MAX_ORDER + 1;

__device__ __forceinline__ double ipow(double b, int e) {
    double r = 1.0;
    for (int i = 0; i < e; ++i) r *= b;
    return r;
}

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Add iv to the int at shared address a + OFF (one instruction, no result wanted).
template <int OFF>
__device__ __forceinline__ void red_shared_add(unsigned a, int iv) {
    asm volatile("red.shared.add.s32 [%0+%1], %2;" : : "r"(a), "n"(OFF), "r"(iv) : "memory");
}

// Bytes of dynamic shared memory of a CTA of `threads` threads for responses of L taps.
__host__ __device__ constexpr size_t rir_smem_bytes(int threads, int L) {
    return sizeof(double) * 3 * AX + sizeof(float) * 3 * AX + 5 * sizeof(float) * threads +
           sizeof(float) * (size_t)((L + 3) & ~3);
}

constexpr float HEADROOM_LOG2 = 6.f;   // full scale = 2^6 times the direct-path amplitude

// Entries of a warp's ring, each an array of 32: first sample of the window, phi, P0, P1, P2.
enum Ring { R_N = 0, R_PHI = 32, R_P0 = 64, R_P1 = 96, R_P2 = 128, RING = 160 };

// round(v) by additions (the conversion instruction shares the quarter-rate pipe with the
// reciprocals): adding 1.5 2^23 leaves the nearest integer, |v| < 2^22, in the low bits.
constexpr float TO_INT = 12582912.f;
constexpr int INT_BITS = 0x4B400000;
// Images as loud as the direct path reach 2^25 steps: multiples of 16 first, then the rest.
__device__ __forceinline__ int2 round_strong(fftpair::u64 v) {
    using namespace fftpair;
    const u64 m = both(TO_INT);
    const u64 t = fma2(v, both(0.0625f), m);
    const u64 rest = add2(fma2(sub2(m, t), both(16.f), v), m);
    const float2 hi = unpack(t), lo = unpack(rest);
    // (unsigned: sixteen times the bits exceeds 32 of them, and the excess cancels)
    constexpr unsigned BITS = 17u * (unsigned)INT_BITS;
    return make_int2((int)(16u * __float_as_uint(hi.x) + __float_as_uint(lo.x) - BITS),
                     (int)(16u * __float_as_uint(hi.y) + __float_as_uint(lo.y) - BITS));
}

// sin(pi x) / pi, 0 <= x <= 1: the Taylor series up to x^13 on the nearer half (rest below 1e-9)
__device__ __forceinline__ float sin_pi_over_pi(float x) {
    const float y = fminf(x, 1.f - x), z = y * y;
    float p = 1.48428793e-4f;
    p = fmaf(p, z, -2.34608099e-3f);
    p = fmaf(p, z, 2.61478478e-2f);
    p = fmaf(p, z, -0.190751824f);
    p = fmaf(p, z, 0.811742425f);
    p = fmaf(p, z, -1.64493407f);
    return fmaf(p * z, y, y);
}

// The window's half width: below 40, where every tap takes the reciprocal form, 40 (80 taps), and more (at
// most 96 taps).  A lane's taps are 32 apart: only from half width 40 on are the first and the last of every lane far from
// the image.  (1536 responses of 8192 taps, order 12, before the polynomials and now: half width 16 to 39 162 and 154 us,
// 40 162 and 147, 47 165 and 155.)
enum Width { SHORT, FORTY, WIDE };

// leff, leff_all (aug_pipeline, else NULL): where each response ends ([utt][source]: taps up to the last
// non-zero one, 0 for silence) and the largest of all; what lies behind a response's end, and the places of sources
// that there are not, stay as they are then.
template <Width WIDTH, int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS)
rir_image_kernel(const AugUttParams *__restrict__ table, int S_max, int L, int half_w,
                 double fs_over_c, int max_order, int cube, const float *__restrict__ tap_tab, float *__restrict__ rir,
                 int *status, int *leff, int *leff_all) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int *ring = reinterpret_cast<int *>(smem_raw);                 // [THREADS / 32][RING]
    int *h = ring + THREADS / 32 * RING;                           // [L rounded up to 4] fixed-point response
    double *dsq = reinterpret_cast<double *>(h + ((L + 3) & ~3));  // [3][AX] squared coordinate differences
    float *gain = reinterpret_cast<float *>(dsq + 3 * AX);         // [3][AX] wall gains per axis

    const int utt = blockIdx.y, s = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const AugUttParams &row = table[utt];
    float *out = rir + ((int64_t)utt * S_max + s) * L;

    const int n_src = row.n_src, order = row.order;
    int bad = 0;
    if (n_src < 1 || n_src > S_max) bad = aug::R_NSRC;
    else if (order < 0 || order > max_order) bad = aug::R_ORDER;
    if (bad || s >= n_src) {
        if (leff == nullptr)
            for (int i = tid; i < L; i += THREADS) out[i] = 0.f;
        else if (bad == aug::R_ORDER && s < n_src && tid == 0)
            leff[utt * S_max + s] = 0;         // silence
        if (bad && tid == 0 && s == 0) {
            if (atomicCAS(&status[0], -1, utt) == -1) status[1] = bad;
        }
        chain_wait();
        return;
    }

    for (int i = tid; i < ((L + 3) >> 2); i += THREADS) reinterpret_cast<int4 *>(h)[i] = make_int4(0, 0, 0, 0);
    const int side = 2 * order + 1;
    if (tid < 3 * side) {
        const int a = tid / side, k = tid % side - order;
        const int p = k & 1;            // k = 2m - p
        const int m = (k + p) / 2;
        const double img = (1 - 2 * p) * (double)row.src_pos[s][a] + 2.0 * m * (double)row.room[a];
        const double diff = img - (double)row.mic[a];
        dsq[a * AX + k + order] = diff * diff;
        gain[a * AX + k + order] = (float)(ipow((double)row.beta[2 * a], abs(m - p)) *
                                           ipow((double)row.beta[2 * a + 1], abs(m)));
    }
    __syncthreads();
    // images in the slabs of radius 0 .. n - 1 of the lattice's lower half: n (2 n^2 + 1) / 3
    const int lower = (order + 1) * (2 * (order + 1) * (order + 1) + 1) / 3;
    const int total = cube ? side * side * side : lower + order * (2 * order * order + 1) / 3;
    // fixed-point scale: a power of two with 2^31 / scale >= 2^HEADROOM_LOG2 / d0
    const float d0sq = (float)(dsq[order] + dsq[AX + order] + dsq[2 * AX + order]);
    const float e2 = d0sq > 0.f ? floorf(31.f - HEADROOM_LOG2 + 0.5f * log2f(d0sq)) : 0.f;
    const float scale = exp2f(fminf(fmaxf(e2, -60.f), 60.f)), inv_scale = exp2f(-fminf(fmaxf(e2, -60.f), 60.f));

    // Per-lane tap constants, see rir_tap_table.
    using fftpair::u64;
    constexpr bool POLY = WIDTH != SHORT;
    constexpr int REST = WIDTH == WIDE ? 4 : 3;          // degree for the last taps
    const float fhw = (float)half_w;
    const float sgn = ((lane - half_w + 1) & 1) ? -1.f : 1.f;
    float fj[3], cj[3], sj[3], head[5], rest[REST + 1];
    if constexpr (POLY) {
        fj[1] = __ldg(tap_tab + lane);
        cj[1] = __ldg(tap_tab + 32 + lane);
        sj[1] = __ldg(tap_tab + 64 + lane);
#pragma unroll
        for (int i = 0; i < 5; ++i) head[i] = __ldg(tap_tab + 32 * (3 + i) + lane);
#pragma unroll
        for (int i = 0; i <= REST; ++i) rest[i] = __ldg(tap_tab + 32 * (8 + i) + lane);
    } else {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            fj[i] = __ldg(tap_tab + 32 * (3 * i) + lane);
            cj[i] = __ldg(tap_tab + 32 * (3 * i + 1) + lane);
            sj[i] = __ldg(tap_tab + 32 * (3 * i + 2) + lane);
        }
    }
    const u64 nsgn = fftpair::both(-sgn);
    const float hann = 3.14159265358979323846f / fhw;
    const double tau_end = (double)(L + half_w - 1);     // windows of later images begin behind the buffer
    constexpr int NW = THREADS / 32;
    const unsigned h_addr = (unsigned)__cvta_generic_to_shared(h) + 4u * lane;
    const unsigned h_rest = h_addr + (lane < 16 ? 256u : 192u);      // of this lane's tap among the last 16
    // first-tap samples for which all 96 lane slots (80 of them taps) stay inside the response
    const unsigned inside = (unsigned)max(L - 96, 0);
    int *my = ring + warp * RING;

    for (int base = warp * 32; base < total; base += NW * 32) {
        // ---- phase A: one image per lane
        const int idx = base + lane;
        bool valid = idx < total;
        int n_first = 0;
        bool strong = false;
        float phi = 0.5f, p0 = 0.f, p1 = 0.f, p2 = 0.f;
        if (valid) {
            int ix, ky, kz;
            if (cube) {
                ix = idx / (side * side);
                const int rem = idx - ix * side * side;
                ky = rem / side - order;
                kz = rem % side - order;
            } else {
                // The upper half of the lattice mirrors the lower one.  Radius of the slab: the largest r with
                // r (2 r^2 + 1) / 3 <= qq; cbrt(1.5 qq) is above it by less than one
                const bool up = idx >= lower;
                int qq = up ? total - 1 - idx : idx;
                int r = (int)exp2f(__log2f(1.5f * (float)qq) * (1.f / 3.f));
                if (r * (2 * r * r + 1) > 3 * qq) --r;
                ix = up ? 2 * order - r : r;
                qq -= r * (2 * r * r + 1) / 3;        // position inside the diamond of radius r
                // rows ky = -r..0 hold 1, 3, .., 2r+1 points (qq < (r+1)^2, row u has u^2 before it);
                // rows ky = 1..r mirror rows r-1..0, counted from the end.
                const bool upper = qq >= (r + 1) * (r + 1);
                if (upper) qq = 2 * r * r + 2 * r - qq;
                const int u = (int)sqrtf((float)qq + 0.5f);      // (away from whole numbers)
                ky = upper ? r - u : u - r;
                kz = qq - u * u - u;
            }
            const int iy = ky + order, iz = kz + order;
            const double d2 = dsq[ix] + dsq[AX + iy] + dsq[2 * AX + iz];
            const float g = gain[ix] * gain[AX + iy] * gain[2 * AX + iz];
            const float r0 = rsqrtf((float)d2);
            double e;
            const double tau = image_distance(d2, r0, e) * fs_over_c;
            // its whole part (rounded down): adding 1.5 2^52 leaves the nearest integer in the low word
            const double m = (tau - 0.5) + 6755399441055744.0;
            int n0 = __double2loint(m);
            phi = (float)(tau - (m - 6755399441055744.0));
            if (phi >= 1.f) {                  // rounded up to the next sample
                ++n0;
                phi = 0.f;
            }
            // a fraction of exactly zero would make the centre tap 0/0: 1e-7 of a sample
            // away from it the tap is the same to 3e-7 of its size
            phi = fmaxf(phi, 1e-7f);
            n_first = n0 - half_w + 1;
            const float A = g * fmaf(r0, 0.5f * (float)e, r0);
            valid = d2 > 0.0 && A != 0.f && tau < tau_end;
            // no tap is larger than A
            strong = fabsf(A) * scale >= 4194303.f;
            p0 = -0.5f * A * scale * sin_pi_over_pi(phi);
            float sps, cps;
            if constexpr (POLY) {
                // pi phi / W_h <= 0.08: the series' next terms are below 1e-9
                const float x = phi * hann, z = x * x;
                cps = fmaf(z, fmaf(z, 1.f / 24.f, -0.5f), 1.f);
                sps = fmaf(x * z, fmaf(z, 1.f / 120.f, -1.f / 6.f), x);
            } else {
                sincospif(phi / fhw, &sps, &cps);
            }
            p1 = p0 * cps;
            p2 = p0 * sps;
        }
        const bool in = valid && (unsigned)n_first < inside;
        const unsigned below = (1u << lane) - 1u;
        const unsigned m_strong = __ballot_sync(0xffffffffu, in && strong), m_in = __ballot_sync(0xffffffffu, in);
        const unsigned m_valid = __ballot_sync(0xffffffffu, valid);
        const int n_strong = __popc(m_strong), n_in = __popc(m_in), cnt = __popc(m_valid);
        {
            // strong ones, other ones inside, those at the edges, and lanes without an image, which add
            // nothing if they fill up a group of four
            const int pos = in ? (strong ? __popc(m_strong & below) : n_strong + __popc(m_in & ~m_strong & below))
                               : valid ? n_in + __popc(m_valid & ~m_in & below) : cnt + __popc(~m_valid & below);
            if (!valid) {
                n_first = 0;
                phi = 0.5f;
                p0 = p1 = p2 = 0.f;
            }
            my[R_N + pos] = n_first;
            my[R_PHI + pos] = __float_as_int(phi);
            my[R_P0 + pos] = __float_as_int(p0);
            my[R_P1 + pos] = __float_as_int(p1);
            my[R_P2 + pos] = __float_as_int(p2);
        }
        __syncwarp();
        // ---- phase B: the taps of four images over the lanes
        // A sinc(x) hann(x) = (1/x) (-A sin(pi phi)/pi) (-1)^j (1/2 + 1/2 cos(pi x / W_h)), x = j - phi
        using namespace fftpair;
        const int n_fast = inside == 0 ? 0 : cnt == n_in ? (n_in + 3) & ~3 : n_in & ~3;
        const int n_loud = min((n_strong + 3) & ~3, n_fast);
        auto four = [&](int k, auto loud) {
            auto fixed = [&](u64 x, u64 y) {               // the fixed-point values of x y
                if constexpr (decltype(loud)::value) {
                    return round_strong(mul2(x, y));
                } else {
                    const float2 v = unpack(fma2(x, y, both(TO_INT)));
                    return make_int2(__float_as_int(v.x) - INT_BITS, __float_as_int(v.y) - INT_BITS);
                }
            };
            auto taps = [&](u64 ph, u64 q0, u64 q1, u64 q2, int i) {
                const float2 x = unpack(fma2(nsgn, ph, both(fj[i])));
                return fixed(pack(rcp_approx(x.x), rcp_approx(x.y)), fma2(both(sj[i]), q2, fma2(both(cj[i]), q1, q0)));
            };
            auto far = [&](u64 ph, u64 q0, const float *c, int degree) {
                u64 p = both(c[degree]);
#pragma unroll
                for (int i = degree - 1; i >= 0; --i) p = fma2(p, ph, both(c[i]));
                return fixed(p, q0);
            };
            // every tap of the windows falls inside the response: no index checks, the adds of an image
            // go to fixed offsets from one address
            const int4 n = *reinterpret_cast<const int4 *>(my + R_N + k);
            const ulonglong2 ph = *reinterpret_cast<const ulonglong2 *>(my + R_PHI + k);
            const ulonglong2 q0 = *reinterpret_cast<const ulonglong2 *>(my + R_P0 + k);
            const ulonglong2 q1 = *reinterpret_cast<const ulonglong2 *>(my + R_P1 + k);
            const ulonglong2 q2 = *reinterpret_cast<const ulonglong2 *>(my + R_P2 + k);
            const unsigned a = h_addr + 4u * n.x, b = h_addr + 4u * n.y, c = h_addr + 4u * n.z, d = h_addr + 4u * n.w;
            int2 s0, t0;
            if constexpr (POLY) {
                s0 = far(ph.x, q0.x, head, 4);
                t0 = far(ph.y, q0.y, head, 4);
            } else {
                s0 = taps(ph.x, q0.x, q1.x, q2.x, 0);
                t0 = taps(ph.y, q0.y, q1.y, q2.y, 0);
            }
            red_shared_add<0>(a, s0.x);
            red_shared_add<0>(b, s0.y);
            red_shared_add<0>(c, t0.x);
            red_shared_add<0>(d, t0.y);
            const int2 s1 = taps(ph.x, q0.x, q1.x, q2.x, 1), t1 = taps(ph.y, q0.y, q1.y, q2.y, 1);
            red_shared_add<128>(a, s1.x);
            red_shared_add<128>(b, s1.y);
            red_shared_add<128>(c, t1.x);
            red_shared_add<128>(d, t1.y);
            if constexpr (WIDTH == WIDE) {
                const int2 s2 = far(ph.x, q0.x, rest, REST), t2 = far(ph.y, q0.y, rest, REST);
                red_shared_add<256>(a, s2.x);
                red_shared_add<256>(b, s2.y);
                red_shared_add<256>(c, t2.x);
                red_shared_add<256>(d, t2.y);
            } else {
                // the last 16 taps, lower half-warp: first two images, upper half: the others
                const int *w = my + k + 2 * (lane >> 4);
                const int2 m = *reinterpret_cast<const int2 *>(w + R_N);
                const u64 ph2 = *reinterpret_cast<const u64 *>(w + R_PHI), r0 = *reinterpret_cast<const u64 *>(w + R_P0);
                int2 s2;
                if constexpr (POLY)
                    s2 = far(ph2, r0, rest, REST);
                else
                    s2 = taps(ph2, r0, *reinterpret_cast<const u64 *>(w + R_P1), *reinterpret_cast<const u64 *>(w + R_P2), 2);
                red_shared_add<0>(h_rest + 4u * m.x, s2.x);
                red_shared_add<0>(h_rest + 4u * m.y, s2.y);
            }
        };
#pragma unroll 1
        for (int k = 0; k < n_loud; k += 4) four(k, std::true_type());
#pragma unroll 1
        for (int k = n_loud; k < n_fast; k += 4) four(k, std::false_type());
#pragma unroll 1
        for (int w = n_fast; w < cnt; ++w) {
            const int n_f = my[R_N + w];
            const float f = __int_as_float(my[R_PHI + w]), P0 = __int_as_float(my[R_P0 + w]);
            const float P1 = __int_as_float(my[R_P1 + w]), P2 = __int_as_float(my[R_P2 + w]);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int m = n_f + lane + 32 * i;
                float v;
                if (POLY && i != 1) {
                    const float *c = i == 0 ? head : rest;
                    const int degree = i == 0 ? 4 : REST;
                    v = c[degree];
#pragma unroll
                    for (int k = degree - 1; k >= 0; --k) v = fmaf(v, f, c[k]);
                    v *= P0;
                } else {
                    v = rcp_approx(fmaf(-sgn, f, fj[i])) * fmaf(sj[i], P2, fmaf(cj[i], P1, P0));
                }
                const bool mine = WIDTH == WIDE || i < 2 || lane < 16;
                if (mine && (unsigned)m < (unsigned)L) atomicAdd(&h[m], __float2int_rn(v));
            }
        }
        __syncwarp();   // the ring slots are rewritten by the next batch
    }
    __syncthreads();
    chain_next();
    const bool vec = (reinterpret_cast<uintptr_t>(out) & 15) == 0 && (L & 3) == 0;
    int end = L;                               // taps to be written
    if (leff != nullptr) {
        int last = 0;
        for (int i = tid; i < ((L + 3) >> 2); i += THREADS) {
            const int4 q = reinterpret_cast<const int4 *>(h)[i];       // (behind the end of the buffer: zeros)
            if ((q.x | q.y | q.z | q.w) != 0) last = 4 * i + (q.w ? 4 : q.z ? 3 : q.y ? 2 : 1);
        }
        last = __reduce_max_sync(0xffffffffu, last);
        if (lane == 0) ring[warp] = last;
        __syncthreads();
        end = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) end = max(end, ring[w]);
    }
    if (vec) {
        for (int i = tid; i < ((end + 3) >> 2); i += THREADS) {
            const int4 q = reinterpret_cast<const int4 *>(h)[i];
            reinterpret_cast<float4 *>(out)[i] = make_float4((float)q.x * inv_scale, (float)q.y * inv_scale,
                                                             (float)q.z * inv_scale, (float)q.w * inv_scale);
        }
    } else {
        for (int i = tid; i < end; i += THREADS) out[i] = (float)h[i] * inv_scale;
    }
    chain_wait();
    if (leff != nullptr && tid == 0) {
        leff[utt * S_max + s] = end;
        if (leff_all != nullptr) atomicMax(leff_all, end);
    }
}

}  // namespace

// Constants of the taps, a row of 32 lanes each; lane l's taps are jj = l, l + 32 and l + 64 (half width 40 and
// below: 64 + l mod 16), tap jj lies at offset j = jj - W + 1 from n0.  The sign (-1)^j (with that of the sine) is the
// same for all taps of a lane.  Reciprocal form: the signed offset, whose reciprocal is taken, cosine and sine of the
// Hann angle; a tap beyond the window gets an offset so large that its value rounds to zero.  Polynomials: the
// coefficients of (1 + cos(pi (j - phi) / W)) / (j - phi) in powers of phi, which interpolate it at the Chebyshev
// points of 0 <= phi <= 1.  In double, once per context: every warp of the kernel working them out took a tenth of its
// time (4096 x 2 responses of order 8).
//   W < 40   three rows for each of the lane's taps
//   W >= 40  three rows for the middle one, five for the first, five for the last (W = 40: four used)
void rir_tap_table(int W, float *tab) {
    const double PI = 3.14159265358979323846;
    auto reciprocal = [&](int row, int lane, int jj) {
        const int j = jj - W + 1;
        const double sgn = ((lane - W + 1) & 1) ? -1.0 : 1.0;
        tab[32 * row + lane] = jj < 2 * W ? (float)(sgn * j) : 3e18f;
        tab[32 * (row + 1) + lane] = (float)cos(PI * j / W);
        tab[32 * (row + 2) + lane] = (float)sin(PI * j / W);
    };
    auto polynomial = [&](int row, int lane, int jj, int degree) {
        const int j = jj - W + 1, n = degree + 1;
        double x[5], d[5], c[5] = {0, 0, 0, 0, 0};
        for (int i = 0; i < n; ++i) {                       // divided differences, then powers
            x[i] = 0.5 + 0.5 * cos(PI * (2 * i + 1) / (2 * n));
            d[i] = (1.0 + cos(PI * (j - x[i]) / W)) / (j - x[i]);
        }
        for (int k = 1; k < n; ++k)
            for (int i = n - 1; i >= k; --i) d[i] = (d[i] - d[i - 1]) / (x[i] - x[i - k]);
        for (int k = n - 1; k >= 0; --k) {
            for (int i = n - 1; i > 0; --i) c[i] = c[i - 1] - x[k] * c[i];
            c[0] = d[k] - x[k] * c[0];
        }
        const double sgn = jj >= 2 * W ? 0.0 : ((lane - W + 1) & 1) ? -1.0 : 1.0;
        for (int i = 0; i < n; ++i) tab[32 * (row + i) + lane] = (float)(sgn * c[i]);
    };
    for (int lane = 0; lane < 32; ++lane) {
        if (W < 40) {
            for (int i = 0; i < 3; ++i) reciprocal(3 * i, lane, i < 2 ? lane + 32 * i : 64 + (lane & 15));
        } else {
            reciprocal(0, lane, lane + 32);
            polynomial(3, lane, lane, 4);
            polynomial(8, lane, W == 40 ? 64 + (lane & 15) : 64 + lane, W == 40 ? 3 : 4);
        }
    }
}

template <Width WIDTH, int THREADS>
static int launch_rir_kernel(AugCtx *ctx, const AugUttParams *table, int B, float *rir, bool chained) {
    const AugConfig &c = ctx->cfg;
    const size_t smem = rir_smem_bytes(THREADS, c.rir_taps);
    const double fs_over_c = (double)c.fs / (double)c.sound_speed;
    const int cube = c.image_lattice == AUG_LATTICE_CUBE ? 1 : 0;
    dim3 grid(c.max_sources, B);
    auto kern = rir_image_kernel<WIDTH, THREADS>;
    if (smem_opt_in<rir_image_kernel<WIDTH, THREADS>>(ctx->device) != AUG_OK) return AUG_ECUDA;
    if (chained) {
        int *leff_all = ctx->route == aug::ROUTE_STORED ? ctx->counters + aug::LEFF_ALL : nullptr;
        if (launch_chained(kern, grid, THREADS, smem, ctx->stream, table, c.max_sources, c.rir_taps, c.frac_half_width,
                           fs_over_c, c.max_order, cube, ctx->tap_tab, rir, ctx->status, ctx->leff, leff_all) != AUG_OK)
            return AUG_ECUDA;
    } else {
        kern<<<grid, THREADS, smem, ctx->stream>>>(table, c.max_sources, c.rir_taps, c.frac_half_width, fs_over_c,
                                                   c.max_order, cube, ctx->tap_tab, rir, ctx->status, nullptr, nullptr);
        AUG_CUDA_OK(cudaGetLastError());
    }
    ctx->launches++;
    return AUG_OK;
}
template <int THREADS>
static int launch_rir_as(AugCtx *ctx, const AugUttParams *table, int B, float *rir, bool chained) {
    const int w = ctx->cfg.frac_half_width;
    return w < 40    ? launch_rir_kernel<SHORT, THREADS>(ctx, table, B, rir, chained)
           : w == 40 ? launch_rir_kernel<FORTY, THREADS>(ctx, table, B, rir, chained)
                     : launch_rir_kernel<WIDE, THREADS>(ctx, table, B, rir, chained);
}

// Both sizes keep 32 warps with 64 registers on a multiprocessor.  Two CTAs of 512 threads are better
// as long as one round of them does (100 responses of 8192 taps, order 10: 17 us, with four of 256 threads
// 21; long responses fit only twice, 300 of 24000 taps: 56 against 64), four of 256 balance better
// beyond where they fit (300 of 8192 taps, order 6: 16.4 against 14.8, 600 23.1 and 21.0; 1200 of 4096
// taps, order 8: 56 and 52).  How many responses there are depends on the table: at least one an
// utterance, at most max_sources.  With so few
// images that eight warps do them in one pass the first round is mostly set-up, and four CTAs are
// taken as soon as there may be more than one (300 of 1600 taps, order 4: 13.0 against 8.9).
int launch_rir(AugCtx *ctx, const AugUttParams *table, int B, float *rir, bool chained) {
    const AugConfig &c = ctx->cfg;
    const bool fit = 4 * (rir_smem_bytes(256, c.rir_taps) + 1024) <= (size_t)ctx->smem_per_sm;
    const int side = 2 * c.max_order + 1;
    const int images = c.image_lattice == AUG_LATTICE_CUBE ? side * side * side
                                                           : side * (2 * c.max_order * (c.max_order + 1) + 3) / 3;
    const int64_t most = (int64_t)B * c.max_sources, round = 2 * (int64_t)ctx->sm_count;
    const bool many = B > round || most >= 2 * round || (images <= 256 && most > round);
    return fit && many ? launch_rir_as<256>(ctx, table, B, rir, chained) : launch_rir_as<512>(ctx, table, B, rir, chained);
}
