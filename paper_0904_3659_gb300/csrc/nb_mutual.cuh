// nb_mutual.cuh -- the mutual inner loop: every unordered pair of particles is
// evaluated once and its two contributions to Eq. (gravity) (Fujiwara &
// Nakasato, arXiv:0904.3659, Section "Introduction") go to both particles.
//
// The difference d = x_i - x_j, s = |d|^2 + eps^2 and y = s^{-1/2} are shared
// by the two sides:
//     a_i += m_j y^3 d     p_i += m_j y        a_j -= m_i y^3 d     p_j += m_i y
// 16 to 19 FP32 lane-operations (see MutualWeights) and one reciprocal square
// root per unordered pair, against 26 when each ordered pair is evaluated by
// itself.
//
// A warp holds 64 P i-particles (slot k of lane l is particle 32 k + l) and
// meets 32 j-particles at a time. At step t lane l works on particle l ^ t of
// the 32, so every lane has another j; the four sums of a j-particle travel
// from lane to lane with it (one exclusive-or shuffle each per step), so after
// 32 steps each j-particle has met every i-particle of the warp and its sums
// are back in the lane of its own number. The order of every addition is fixed.
//
// What bounds it: the register file. An FP32 instruction reads two registers a
// cycle; a fused multiply-add of three different registers therefore takes 1.5
// cycles unless the compiler can keep one of them in the operand cache
// (measured on sm_103a: 1.5-1.66 scalar, 3.5 packed, against 1.03-1.05 and
// 2.0-2.3 for two-operand instructions). So only the instructions with at most
// two different operands run packed (s, y^2, y^3), the rest scalar. Measured
// with two weights per pair, FP32 pipe busy: all packed 62%, all scalar 66%,
// this mix 71%; 2 warps per scheduler 69%, 3 (at most 168 registers) 71%, 4
// with 4 i-particles each 65%.
#pragma once

#include "nb_device.cuh"

namespace nbk {
using namespace nbdev;

// One particle of the mutual kernels, 16 bytes: (-x, -y, -z, -m/2). In HL form
// (positions from FP64 state, see kHLRecords) two of them: grid parts and
// -m/2, then remainders and 0.
using MPart = float4;

// How a pair's weights are formed, chosen on the device for the whole call:
//  kEqual    every mass has the same bits: the sums are taken without masses
//            (w = y^3 on both sides) and the combine multiplies by the mass: 16
//            operations (14 without the potential).
//  kProduct  w = ((c m_i m_j) y) y^2, one weight for both sides; the combine
//            divides by a particle's own c m_i. 18 operations. c is a power of
//            two (product_scale) that keeps every product and sum inside FP32's
//            range for masses within a factor of the first one and distances up to
//            a multiple of eps that depend on eps (2^28 and 2^34 up to eps = 1, 2^15
//            and 2^21 at eps = 2^40).
//  kWide     w_i = ((-m_j/2) y) y^2, w_j = ((-m_i/2) y) y^2: 19 operations, for
//            everything else (massless particles, wider ranges of masses or
//            distances, positions or softening outside [2^-40, 2^40],
//            infinities and NaN).
// One weight for both sides also means fewer registers read. Measured at N =
// 131072, G-interactions/s: kEqual 3450, kProduct 3090, and 2830-2980 for the
// form w_i = (-m_j/2) y^3, w_j = (-m_i/2) y^3, also 18 operations.
// (kAny, of a kernel: it runs whichever the call needs.)
enum MutualWeights : int { kEqual = 0, kProduct = 1, kWide = 2, kAny = 3 };
constexpr float kMutualRange = 1099511627776.f;  // 2^40

// What a pack block reports about its particles (bits).
enum MutualNote : int { kNoteUnequal = 1, kNoteNoProduct = 2, kNoteWide = 4 };

// The form of the weights for a call whose pack blocks reported `notes`.
__device__ __forceinline__ int mutual_weights(int notes) {
    if (notes & kNoteWide) return kWide;
    if (!(notes & kNoteUnequal)) return kEqual;
    return notes & kNoteNoProduct ? kWide : kProduct;
}

// kProduct's ranges. With e the exponent of eps and e0 that of the first particle's
// -m/2, every -m/2 lies within 2^+-ratio of the first one's, every coordinate within
// 2^(reach - 2) eps, so every distance below 2^reach eps, and c = 2^(shift - 2 e0).
// The products and sums are then bounded by
//   c m_i              2^(t - ratio) .. 2^(t + ratio + 1) with t = shift - e0
//   c m_i m_j          2^(shift - 2 ratio) .. 2^(shift + 2 ratio + 2)
//   c m_i m_j y        2^(shift - e + 2 ratio + 2), 2^31 of them by 2^(shift - e + 2 ratio + 33)
//   w = c m_i m_j y^3  2^(shift - 3 e - 2 ratio - 3 reach - 3) .. 2^(shift - 3 e + 2 ratio + 2)
//   w d                2^(shift - 2 e + 2 ratio + 1), 2^31 of them by 2^(shift - 2 e + 2 ratio + 32)
// For the products to be normal numbers and the sums to be finite, 4 ratio + 3 reach
// may be 214 - max(2 e, 3 e - 33, 0): where eps > 1 masses and distances give up as
// many powers of two each. What room `shift` has goes to the range of the first mass.
struct ProductScale {
    int ratio, reach, shift;
    bool fits;  // c m_i is a normal number
};
__host__ __device__ constexpr ProductScale product_scale(int e0, int e) {
    const auto lesser = [](int a, int b) { return a < b ? a : b; };
    const auto greater = [](int a, int b) { return a > b ? a : b; };
    const int less = (greater(greater(2 * e, 3 * e - 33), 0) + 6) / 7, ratio = 28 - less, reach = 34 - less;
    const int least = greater(3 * e + 2 * ratio + 3 * reach - 122, 2 * ratio - 126);
    const int most = 94 - 2 * ratio + lesser(lesser(e, 2 * e + 1), lesser(3 * e + 31, 31));
    const int shift = greater(least, lesser(e0, most)), t = shift - e0;
    return {ratio, reach, shift, t - ratio >= -126 && t + ratio <= 126};
}

// c m_i of an i-particle's -m_i/2.
__device__ __forceinline__ float mutual_scale(float hm, float hm0, float eps) {
    const int e0 = ilogbf(hm0);
    return ldexpf(hm, product_scale(e0, ilogbf(eps)).shift - 2 * e0);
}

// Padding records: no mass, and so far away that s overflows to infinity and y
// is exactly 0 against any particle within kMutualRange.
__device__ __forceinline__ MPart mutual_padding() { return make_float4(-7.378697629e19f, 0.f, 0.f, 0.f); }  // -2^66

// A block of a pack kernel adds the notes on its particles (v: the record of a
// real particle; hm0: -m/2 of the first particle) to the call's word, which is
// zero between calls. Called by whole blocks.
__device__ __forceinline__ void mutual_note(bool real, const MPart &v, float hm0, float eps, int *notes) {
    int k = 0;
    if (real) {
        const float r = fmaxf(fabsf(v.x), fmaxf(fabsf(v.y), fabsf(v.z))), m = fabsf(v.w), m0 = fabsf(hm0);
        if (!(r <= kMutualRange) || v.x != v.x || v.y != v.y || v.z != v.z) k |= kNoteWide;
        if (__float_as_uint(v.w) != __float_as_uint(hm0) || !(m <= 1.7e38f)) k |= kNoteUnequal;
        const bool normal = m0 >= 1e-37f && m0 <= 1e37f;  // not zero, subnormal, infinite, NaN
        const ProductScale q = product_scale(normal ? ilogbf(hm0) : 0, ilogbf(eps));
        if (!normal || !q.fits || !(r <= ldexpf(eps, q.reach - 2)) ||
            !(m >= ldexpf(m0, -q.ratio) && ldexpf(m, -q.ratio) <= m0))
            k |= kNoteNoProduct;
    }
    const int any = __syncthreads_or(k & kNoteUnequal) * kNoteUnequal |
                    (__syncthreads_or(k & kNoteNoProduct) ? kNoteNoProduct : 0) |
                    (__syncthreads_or(k & kNoteWide) ? kNoteWide : 0);
    if (threadIdx.x == 0 && any) atomicOr(notes, any);
}

// The i-particles of a thread: P packed pairs.
template <int P, bool HL>
struct MutualI {
    float2 x[P], y[P], z[P], hm[P];
    float2 lx[HL ? P : 1], ly[HL ? P : 1], lz[HL ? P : 1];
};

// x_i - x_j of pair q; scalar, see the header comment.
template <int P, bool HL>
__device__ __forceinline__ void mutual_diff(const MutualI<P, HL> &I, int q, const float4 &h,
                                            const float4 &l, float2 &dx, float2 &dy, float2 &dz) {
    dx = make_float2(__fadd_rn(I.x[q].x, h.x), __fadd_rn(I.x[q].y, h.x));
    dy = make_float2(__fadd_rn(I.y[q].x, h.y), __fadd_rn(I.y[q].y, h.y));
    dz = make_float2(__fadd_rn(I.z[q].x, h.z), __fadd_rn(I.z[q].y, h.z));
    if (HL) {
        dx.x = __fadd_rn(dx.x, __fadd_rn(I.lx[q].x, l.x));
        dx.y = __fadd_rn(dx.y, __fadd_rn(I.lx[q].y, l.x));
        dy.x = __fadd_rn(dy.x, __fadd_rn(I.ly[q].x, l.y));
        dy.y = __fadd_rn(dy.y, __fadd_rn(I.ly[q].y, l.y));
        dz.x = __fadd_rn(dz.x, __fadd_rn(I.lz[q].x, l.z));
        dz.y = __fadd_rn(dz.y, __fadd_rn(I.lz[q].y, l.z));
    }
}

// A sum S + E with the factor that its weights left out, in one rounding: f = -m/2
// of all masses (kEqual), c m_i (kProduct).
__device__ __forceinline__ float mutual_result(int weights, float S, float E, float f) {
    const float s = -2.f * S, e = -2.f * E;
    if (weights == kEqual) {
        const float p = __fmul_rn(s, f);
        const float v = __fadd_rn(p, __fmaf_rn(e, f, __fmaf_rn(s, f, -p)));
        return isfinite(v) ? v : __fmul_rn(__fadd_rn(s, e), f);
    }
    if (weights == kProduct) {
        const float q = __fdiv_rn(s, f);
        const float v = __fadd_rn(q, __fdiv_rn(__fadd_rn(__fmaf_rn(-q, f, s), e), f));
        return isfinite(v) ? v : __fdiv_rn(__fadd_rn(s, e), f);
    }
    return __fadd_rn(s, e);
}

// One group of 32 j-particles T[0..31] (HL: T[2k], T[2k + 1]) against the
// warp's i-particles. With w the weights above, acc[q][0..2] += w_i d and
// acc[q][3] += w_i s, and on return ja[0..2] = sum w_j d and ja[3] = sum w_j s
// over the warp's i-particles for j-particle `lane` (w s: the weight before its
// factor y^2, that is (-m/2) y, c m_i m_j y or y). On FP64 state the j-side sums
// are taken in runs of RUN steps, 16 P RUN terms, whose totals travel apart: the
// error of a against FP64 6.6e-8 -> 6.0e-8 (N = 20011, 256 terms before) at the
// same time (1397 -> 1398 us for four steps and the energy; 1.0e-7 -> 9.9e-8 and
// 611 -> 615 us for 300 clusters).
template <int P, int UNR, bool POT, bool HL, int W>
__device__ __forceinline__ void mutual_group(const MPart *__restrict__ T, int lane,
                                             const MutualI<P, HL> &I, float2 (&acc)[P][4],
                                             float (&ja)[4], const float2 eps2) {
#pragma unroll
    for (int c = 0; c < 4; ++c) ja[c] = 0.f;
    constexpr int RUN = HL ? 8 : 32;
    float jt[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int t0 = 0; t0 < 32; t0 += RUN) {
#pragma unroll UNR
        for (int t1 = 0; t1 < RUN; ++t1) {
            const int t = t0 + t1;
            const int k = lane ^ t;
            const float4 h = T[HL ? 2 * k : k];
            const float4 l = HL ? T[2 * k + 1] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int q = 0; q < P; ++q) {
                float2 dx, dy, dz;
                mutual_diff<P, HL>(I, q, h, l, dx, dy, dz);
                float2 s = fma2(dx, dx, eps2);
                s = fma2(dy, dy, s);
                s = fma2(dz, dz, s);
                const float2 y = make_float2(rsqrt_sfu(s.x), rsqrt_sfu(s.y));
                const float2 y2 = mul2(y, y);
                float2 wi, wj, pi, pj;
                if (W == kEqual) {
                    pi = pj = y;
                    wi = wj = mul2(y2, y);
                } else if (W == kProduct) {
                    pi = pj = make_float2(__fmul_rn(__fmul_rn(I.hm[q].x, h.w), y.x),
                                          __fmul_rn(__fmul_rn(I.hm[q].y, h.w), y.y));
                    wi = wj = make_float2(__fmul_rn(pi.x, y2.x), __fmul_rn(pi.y, y2.y));
                } else {
                    pi = make_float2(__fmul_rn(h.w, y.x), __fmul_rn(h.w, y.y));
                    pj = make_float2(__fmul_rn(I.hm[q].x, y.x), __fmul_rn(I.hm[q].y, y.y));
                    wi = make_float2(__fmul_rn(pi.x, y2.x), __fmul_rn(pi.y, y2.y));
                    wj = make_float2(__fmul_rn(pj.x, y2.x), __fmul_rn(pj.y, y2.y));
                }
                acc[q][0] = make_float2(__fmaf_rn(wi.x, dx.x, acc[q][0].x), __fmaf_rn(wi.y, dx.y, acc[q][0].y));
                acc[q][1] = make_float2(__fmaf_rn(wi.x, dy.x, acc[q][1].x), __fmaf_rn(wi.y, dy.y, acc[q][1].y));
                acc[q][2] = make_float2(__fmaf_rn(wi.x, dz.x, acc[q][2].x), __fmaf_rn(wi.y, dz.y, acc[q][2].y));
                ja[0] = __fmaf_rn(wj.x, dx.x, ja[0]);
                ja[1] = __fmaf_rn(wj.x, dy.x, ja[1]);
                ja[2] = __fmaf_rn(wj.x, dz.x, ja[2]);
                ja[0] = __fmaf_rn(wj.y, dx.y, ja[0]);
                ja[1] = __fmaf_rn(wj.y, dy.y, ja[1]);
                ja[2] = __fmaf_rn(wj.y, dz.y, ja[2]);
                if (POT) {
                    acc[q][3] = W == kEqual ? add2(acc[q][3], pi)
                                            : make_float2(__fadd_rn(acc[q][3].x, pi.x), __fadd_rn(acc[q][3].y, pi.y));
                    ja[3] = __fadd_rn(ja[3], pj.x);
                    ja[3] = __fadd_rn(ja[3], pj.y);
                }
            }
            // The sums move on with their particle: particle j is at lane j ^ t
            // now and at lane j ^ (t + 1) next (after the last step, at home).
            const int move = (t ^ (t + 1)) & 31;
#pragma unroll
            for (int c = 0; c < (POT ? 4 : 3); ++c) ja[c] = __shfl_xor_sync(0xffffffffu, ja[c], move);
        }
        if (RUN < 32) {
            const int move = (t0 ^ (t0 + RUN)) & 31;
#pragma unroll
            for (int c = 0; c < (POT ? 4 : 3); ++c) {
                jt[c] = __fadd_rn(__shfl_xor_sync(0xffffffffu, jt[c], move), ja[c]);
                ja[c] = 0.f;
            }
        }
    }
    if (RUN < 32)
#pragma unroll
        for (int c = 0; c < (POT ? 4 : 3); ++c) ja[c] = jt[c];
}

// A group of the warp's own particles, i-slot `self` of each lane, for the
// i-side alone (both orders of these pairs are met this way): every lane reads
// the same j, and slot `self` of lane l leaves out particle l.
template <int P, bool POT, bool HL, int W>
__device__ __forceinline__ void self_group(const MPart *__restrict__ T, int lane, int self,
                                           const MutualI<P, HL> &I, float2 (&acc)[P][4],
                                           const float2 eps2) {
#pragma unroll 1
    for (int t = 0; t < 32; ++t) {
        const float4 h = T[HL ? 2 * t : t];
        const float4 l = HL ? T[2 * t + 1] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < P; ++q) {
            float2 dx, dy, dz;
            mutual_diff<P, HL>(I, q, h, l, dx, dy, dz);
            float2 s = fma2(dx, dx, eps2);
            s = fma2(dy, dy, s);
            s = fma2(dz, dz, s);
            const float2 y = make_float2(rsqrt_sfu(s.x), rsqrt_sfu(s.y));
            float2 m = splat2(h.w);
            if (W == kProduct) m = mul2(I.hm[q], m);
            if (W == kEqual) m = y;  // the factor that the self term leaves out
            if (self == 2 * q && t == lane) m.x = 0.f;
            if (self == 2 * q + 1 && t == lane) m.y = 0.f;
            const float2 p = W == kEqual ? m : mul2(m, y);
            if (POT) acc[q][3] = add2(acc[q][3], p);
            const float2 w = mul2(p, mul2(y, y));
            acc[q][0] = fma2(w, dx, acc[q][0]);
            acc[q][1] = fma2(w, dy, acc[q][1]);
            acc[q][2] = fma2(w, dz, acc[q][2]);
        }
    }
}

// The group functions for the kernel's form of the weights. With massless particles
// (kWide) a kAny kernel unrolled once was slower than the direct kernels: nb_force N =
// 13312 89.4 us and with UNR = 4 85.1 (stream-K form 85.0), N = 16896 135 and 127 (133),
// 1024 clusters up to 4096 830 and 795; equal masses 1% more. On two-word positions once
// is fast enough (300 clusters 131 us a step; 145 for the direct kernels), and 4 costs
// equal masses 1%.
template <int P, int UNR, bool POT, bool HL, int W>
__device__ __forceinline__ void run_group(int weights, const MPart *G, int lane, const MutualI<P, HL> &I,
                                          float2 (&acc)[P][4], float (&ja)[4], float2 eps2) {
    if constexpr (W != kAny)
        mutual_group<P, UNR, POT, HL, W>(G, lane, I, acc, ja, eps2);
    else if (weights == kEqual)
        mutual_group<P, UNR, POT, HL, kEqual>(G, lane, I, acc, ja, eps2);
    else if (weights == kProduct)
        mutual_group<P, UNR, POT, HL, kProduct>(G, lane, I, acc, ja, eps2);
    else
        mutual_group<P, (HL ? 1 : UNR), POT, HL, kWide>(G, lane, I, acc, ja, eps2);
}

template <int P, bool POT, bool HL, int W>
__device__ __forceinline__ void run_self(int weights, const MPart *G, int lane, int self, const MutualI<P, HL> &I,
                                         float2 (&acc)[P][4], float2 eps2) {
    if constexpr (W != kAny)
        self_group<P, POT, HL, W>(G, lane, self, I, acc, eps2);
    else if (weights == kEqual)
        self_group<P, POT, HL, kEqual>(G, lane, self, I, acc, eps2);
    else if (weights == kProduct)
        self_group<P, POT, HL, kProduct>(G, lane, self, I, acc, eps2);
    else
        self_group<P, POT, HL, kWide>(G, lane, self, I, acc, eps2);
}

}  // namespace nbk
