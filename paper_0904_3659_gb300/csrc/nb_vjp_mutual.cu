// nb_vjp_mutual.cu -- the vector-Jacobian product of Eq. (gravity) (nb_vjp.cu has
// the formulas) with every unordered pair evaluated once, in the manner of
// nb_mutual.cu: the same triangle of (i-block, j-tile) units, the j-side sums
// travelling through the lanes with their particle, the same combine.
//
// For a pair (i, l), r = x_i - x_l, y = (|r|^2 + eps^2)^{-1/2}, with the scalar
// products s_i = r.ga_i and s_l = r.ga_l, the coefficient of r is the same for
// both particles:
//   c = 3 y^3 [ m_i (y^2 s_l - gp_l / 3) - m_l (y^2 s_i + gp_i / 3) ]
//   R_i += c r         R_l -= c r
//   S_i += m_l y^3     S_l += m_i y^3
//   V_i += y^3 ga_l    V_l += y^3 ga_i
//   G_i += gp_l y - s_l y^3     G_l += gp_i y + s_i y^3
// and gx = R + ga S - m V, gm = G. 37 FP32 operations and one reciprocal square
// root per unordered pair (34 without gp), against 56 (52) when each ordered pair
// is evaluated by itself. The masses enter last: y^2 s is of the order of the gradient
// over a distance, whereas m s overflows FP32 in units of metres and kilograms. The
// records hold gp / 3 and the factor 3 of c is the combine's. (Without gp the direct
// kernel forms m s too, c = y^3 y^2 (3 m_i s_l - 3 m_l s_i), and so does this one.)
#include <algorithm>

#include "nb_device.cuh"
#include "nb_ext.h"
#include "nb_internal.h"
#include "nb_triangle.cuh"

namespace nbk {
using namespace nbdev;

// One particle: (-x, -y, -z, m), (ga_x, ga_y, ga_z, gp / 3). Padding is all zero:
// without m, ga and gp a particle adds nothing to others.
constexpr int kVmRecords = 2;

__global__ void vjp_mutual_pack_kernel(const float *__restrict__ x, const float *__restrict__ m,
                                       const float *__restrict__ ga, const float *__restrict__ gp, int64_t n,
                                       int64_t npad, float4 *__restrict__ cp) {
    pdl_wait_then_release();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= npad) return;
    float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u;
    if (i < n) {
        u = make_float4(-x[3 * i], -x[3 * i + 1], -x[3 * i + 2], m[i]);
        v = make_float4(ga[3 * i], ga[3 * i + 1], ga[3 * i + 2], gp ? __fdiv_rn(gp[i], 3.f) : 0.f);
    }
    cp[kVmRecords * i] = u;
    cp[kVmRecords * i + 1] = v;
}

// The same from the leap-frog adjoint's state.
__global__ void vjp_mutual_pack_state_kernel(const nbx::VjpState s, const float *__restrict__ m, int64_t n,
                                             int64_t npad, float4 *__restrict__ cp) {
    pdl_wait_then_release();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= npad) return;
    float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u;
    if (i < n) {
        float x[3], g[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double l = s.la[3 * i + c];
            x[c] = (float)s.x[3 * i + c];
            g[c] = (float)(s.first ? l : l + (-((0.5 * s.dt) * s.lv[3 * i + c])));
        }
        u = make_float4(-x[0], -x[1], -x[2], m[i]);
        v = make_float4(g[0], g[1], g[2], 0.f);
    }
    cp[kVmRecords * i] = u;
    cp[kVmRecords * i + 1] = v;
}

struct VmArgs {
    const float4 *cp;      // [npad][2]
    float4 *pi;            // [grid + rows][4][ib]: sums (R, S), (V, G), their carries
    float4 *pj;            // [entry][2]: j-side (R, S), (V, G)
    int *row_first, *row_last;
    int *err;
    int64_t njt, nib, r0, r1, tiles;
    int grid;
    float eps2;
    int64_t fault_unit;
    uint64_t wait_ns;
    int64_t npad, pi_len, pj_len;
};

struct VmOut {
    float *gx, *gm;
    nbx::VjpState adj;     // (adj.lx: the results go there)
    float4 *state;         // [n][4] sums and carries between panels
    int64_t n;
    int ib, jt, last;
    float r_factor;        // of the sums of R
};

// The i-particles of a thread: P packed pairs.
template <int P>
struct VmI {
    float2 x[P], y[P], z[P], m[P], m3[P], gx[P], gy[P], gz[P], gp[P];
};

// One half of a packed pair against one l; a: the sums of i, b: those of l.
// Eight sums, and with GP a ninth: the two parts of G, sum s y^3 and sum (gp / 3) y, stay
// apart over a run of additions, because each addition to the larger rounds
// (relative error of gm against FP64, N = 8192: 3.2e-7 in one sum, 2.3e-7 in two, 2.4e-7
// the direct kernel).
template <bool GP>
constexpr int kVmSums = GP ? 9 : 8;

template <bool GP, bool BOTH>
__device__ __forceinline__ void vm_pair(float dx, float dy, float dz, float y, float y2, float y3, float mi, float m3i,
                                        float gix, float giy, float giz, float gpi, const float4 &h, const float4 &g,
                                        float m3l, float *(&a)[kVmSums<GP>], float (&b)[kVmSums<GP>]) {
    const float si = __fmaf_rn(dz, giz, __fmaf_rn(dy, giy, __fmul_rn(dx, gix)));
    const float sl = __fmaf_rn(dz, g.z, __fmaf_rn(dy, g.y, __fmul_rn(dx, g.x)));
    float t;  // GP: without the factor 3
    if (GP) t = __fmaf_rn(-h.w, __fmaf_rn(y2, si, gpi), __fmul_rn(mi, __fmaf_rn(y2, sl, -g.w)));
    else t = __fmul_rn(y2, __fmaf_rn(-m3l, si, __fmul_rn(m3i, sl)));
    const float c = __fmul_rn(y3, t);
    *a[0] = __fmaf_rn(c, dx, *a[0]);
    *a[1] = __fmaf_rn(c, dy, *a[1]);
    *a[2] = __fmaf_rn(c, dz, *a[2]);
    *a[3] = __fmaf_rn(h.w, y3, *a[3]);
    *a[4] = __fmaf_rn(y3, g.x, *a[4]);
    *a[5] = __fmaf_rn(y3, g.y, *a[5]);
    *a[6] = __fmaf_rn(y3, g.z, *a[6]);
    *a[7] = __fmaf_rn(-sl, y3, *a[7]);
    if constexpr (GP) *a[8] = __fmaf_rn(g.w, y, *a[8]);
    if (BOTH) {  // b[0..2] holds -R_l
        b[0] = __fmaf_rn(c, dx, b[0]);
        b[1] = __fmaf_rn(c, dy, b[1]);
        b[2] = __fmaf_rn(c, dz, b[2]);
        b[3] = __fmaf_rn(mi, y3, b[3]);
        b[4] = __fmaf_rn(y3, gix, b[4]);
        b[5] = __fmaf_rn(y3, giy, b[5]);
        b[6] = __fmaf_rn(y3, giz, b[6]);
        b[7] = __fmaf_rn(si, y3, b[7]);
        if constexpr (GP) b[8] = __fmaf_rn(gpi, y, b[8]);
    }
}

// 32 particles T[2k], T[2k + 1] against the warp's i-particles (BOTH: for both
// sides, lane l meeting particle l ^ t at step t; else for the i-side alone, all
// lanes meeting particle t, and slot `self` of lane l leaving out particle l). The
// sums of l are taken in runs of RUN steps, 2 P RUN terms, whose totals travel apart.
template <int P, int UNR, bool GP, bool BOTH, int RUN>
__device__ __forceinline__ void vm_group(const float4 *__restrict__ T, int lane, int self, const VmI<P> &I,
                                         float2 (&acc)[P][kVmSums<GP>], float (&b)[kVmSums<GP>], const float2 eps2) {
    float bt[kVmSums<GP>] = {};
#pragma unroll 1
    for (int t0 = 0; t0 < 32; t0 += RUN) {
#pragma unroll UNR
        for (int t1 = 0; t1 < RUN; ++t1) {
            const int t = t0 + t1;
            const int k = BOTH ? lane ^ t : t;
            const float4 h = T[kVmRecords * k], g = T[kVmRecords * k + 1];
            const float m3l = GP ? 0.f : __fmul_rn(3.f, h.w);
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const float2 dx = make_float2(__fadd_rn(I.x[q].x, h.x), __fadd_rn(I.x[q].y, h.x));
                const float2 dy = make_float2(__fadd_rn(I.y[q].x, h.y), __fadd_rn(I.y[q].y, h.y));
                const float2 dz = make_float2(__fadd_rn(I.z[q].x, h.z), __fadd_rn(I.z[q].y, h.z));
                float2 s = fma2(dx, dx, eps2);
                s = fma2(dy, dy, s);
                s = fma2(dz, dz, s);
                float2 y = make_float2(rsqrt_sfu(s.x), rsqrt_sfu(s.y));
                if (!BOTH) {
                    if (self == 2 * q && t == lane) y.x = 0.f;
                    if (self == 2 * q + 1 && t == lane) y.y = 0.f;
                }
                const float2 y2 = mul2(y, y), y3 = mul2(y2, y);
                float *ax[kVmSums<GP>], *ay[kVmSums<GP>];
#pragma unroll
                for (int c = 0; c < kVmSums<GP>; ++c) {
                    ax[c] = &acc[q][c].x;
                    ay[c] = &acc[q][c].y;
                }
                vm_pair<GP, BOTH>(dx.x, dy.x, dz.x, y.x, y2.x, y3.x, I.m[q].x, I.m3[q].x, I.gx[q].x, I.gy[q].x,
                                  I.gz[q].x, I.gp[q].x, h, g, m3l, ax, b);
                vm_pair<GP, BOTH>(dx.y, dy.y, dz.y, y.y, y2.y, y3.y, I.m[q].y, I.m3[q].y, I.gx[q].y, I.gy[q].y,
                                  I.gz[q].y, I.gp[q].y, h, g, m3l, ay, b);
            }
            if (BOTH) {
                const int move = (t ^ (t + 1)) & 31;
#pragma unroll
                for (int c = 0; c < kVmSums<GP>; ++c) b[c] = __shfl_xor_sync(0xffffffffu, b[c], move);
            }
        }
            if (RUN < 32) {
            const int move = (t0 ^ (t0 + RUN)) & 31;
#pragma unroll
            for (int c = 0; c < kVmSums<GP>; ++c) {
                bt[c] = __fadd_rn(__shfl_xor_sync(0xffffffffu, bt[c], move), b[c]);
                b[c] = 0.f;
            }
        }
    }
    if (RUN < 32)
#pragma unroll
        for (int c = 0; c < kVmSums<GP>; ++c) b[c] = bt[c];
}

// As mutual_kernel (nb_mutual.cu), with two records and eight sums per particle. FOLD:
// groups of 32 l between two compensated additions.
template <int WARPS, int P, int JT, int STAGES, int UNR, int MINB, bool GP, int RUN, int FOLD>
__global__ void __launch_bounds__(WARPS * 32, MINB) vjp_mutual_kernel(const VmArgs A) {
    constexpr int THREADS = WARPS * 32;
    constexpr int IB = 64 * P * WARPS;
    constexpr int TPB = IB / JT;
    constexpr uint32_t TILE_BYTES = JT * kVmRecords * sizeof(float4);
    constexpr bool FOLD_IN_TILE = FOLD * 32 < JT;
    static_assert(FOLD_IN_TILE || FOLD * 32 % JT == 0, "a fold ends a group or a tile");
    static_assert(IB % JT == 0 && JT % 32 == 0, "whole tiles per block, whole groups per tile");

    // Shared memory: [STAGES tiles][2 x WARPS x JT x 2 j-side sums][running sums,
    // carries][barriers][issue records]
    extern __shared__ __align__(128) unsigned char smem[];
    float4 *tiles = reinterpret_cast<float4 *>(smem);
    float4 *jsum = reinterpret_cast<float4 *>(smem + (size_t)STAGES * TILE_BYTES);
    float2 *ssum = reinterpret_cast<float2 *>(jsum + 2 * WARPS * JT * 2);
    float2 *scmp = ssum + 8 * P * THREADS;
    uint64_t *full = reinterpret_cast<uint64_t *>(scmp + 8 * P * THREADS);
    int *issued_at = reinterpret_cast<int *>(full + STAGES);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t c = blockIdx.x;
    const Triangle T{A.njt, A.nib, TPB};
    const int64_t u0 = c * A.tiles / A.grid, first = T.lin(A.r0) + u0;
    const int count = (int)((c + 1) * A.tiles / A.grid - u0);
    int64_t b, t;
    T.locate(u0, A.r0, A.r1, &b, &t);

    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            issued_at[s] = -1;
        }
        fence_mbar_init();
    }
    __syncthreads();
    pdl_wait();  // (no release: the combine's blocks, resident early, cost 1-2%)

    int64_t pb = b, pt = t;  // thread 0: the next tile to copy
    auto issue = [&](int kk) {
        const int64_t tile = pt;
        if (++pt == A.njt) {
            ++pb;
            pt = pb * TPB;
        }
        if (first + kk == A.fault_unit) return;  // test hook: this copy never happens
        if (!NB_IN(A.err, 50, (tile + 1) * JT <= A.npad)) return;
        const int s = kk % STAGES;
        issued_at[s] = kk;
        mbar_arrive_expect_tx(&full[s], TILE_BYTES);
        bulk_g2s(tiles + (size_t)s * JT * kVmRecords, A.cp + tile * JT * kVmRecords, TILE_BYTES, &full[s]);
    };
    if (tid == 0)
        for (int kk = 0; kk < count && kk < STAGES - 1; ++kk) issue(kk);

    const float2 eps2 = splat2(A.eps2), zero2 = splat2(0.f);
    VmI<P> I;
    float2 acc[P][kVmSums<GP>];
#pragma unroll
    for (int q = 0; q < P; ++q)
#pragma unroll
        for (int r = 0; r < kVmSums<GP>; ++r) acc[q][r] = zero2;
    int held = 0;

    auto fold = [&]() {
#pragma unroll
        for (int q = 0; q < P; ++q) {
            if constexpr (GP) {
                acc[q][7] = fma2(splat2(3.f), acc[q][8], acc[q][7]);
                acc[q][8] = zero2;
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int k = (8 * q + r) * THREADS + tid;
                const float2 s0 = ssum[k];
                const float2 y = add2(acc[q][r], neg2(scmp[k]));
                const float2 v = add2(s0, y);
                scmp[k] = add2(add2(v, neg2(s0)), neg2(y));
                ssum[k] = v;
                acc[q][r] = zero2;
            }
        }
        held = 0;
    };
    auto flush = [&](int64_t row) {
        fold();
        const int64_t off = (c + row - A.r0) * 4 * (int64_t)IB;
        if (!NB_IN(A.err, 51, off >= 0 && off + 4 * IB <= A.pi_len)) return;
        float4 *dst = A.pi + off + warp * 64 * P + lane;
#pragma unroll
        for (int q = 0; q < P; ++q)
#pragma unroll
            for (int w = 0; w < 4; ++w) {  // (R, S), (V, G), their carries
                const float2 *src = (w < 2 ? ssum : scmp) + (8 * q + 4 * (w & 1)) * THREADS + tid;
                const float2 s0 = src[0], s1 = src[THREADS], s2 = src[2 * THREADS], s3 = src[3 * THREADS];
                dst[w * IB + 64 * q] = make_float4(s0.x, s1.x, s2.x, s3.x);
                dst[w * IB + 64 * q + 32] = make_float4(s0.y, s1.y, s2.y, s3.y);
            }
    };
    int64_t put_at = 0;
    auto put = [&](int buf) {
        if (!NB_IN(A.err, 52, 2 * (put_at + JT) <= A.pj_len)) return;
        for (int j = tid; j < 2 * JT; j += THREADS) {
            float4 v = jsum[buf * WARPS * 2 * JT + j];
#pragma unroll
            for (int w = 1; w < WARPS; ++w) {
                const float4 u = jsum[(buf * WARPS + w) * 2 * JT + j];
                v = make_float4(__fadd_rn(v.x, u.x), __fadd_rn(v.y, u.y), __fadd_rn(v.z, u.z),
                                __fadd_rn(v.w, u.w));
            }
            A.pj[2 * put_at + j] = v;
        }
    };

    const int64_t pj0 = T.lin(A.r0);
    int64_t cur = -1;
    int bad = 0;
    for (int k = 0; k < count; ++k) {
        // Every thread is done with tile k - 1: its stage may be refilled and
        // its j-side sums are complete. A timeout ends the loop for all.
        if (__syncthreads_or(bad)) break;
        if (tid == 0 && k + STAGES - 1 < count) issue(k + STAGES - 1);
        if (k > 0) put((k - 1) & 1);

        if (b != cur) {
            if (cur >= 0) flush(cur);
            cur = b;
            if (tid == 0 && t == b * TPB) A.row_first[b] = (int)c;
#pragma unroll
            for (int q = 0; q < P; ++q) {
                int64_t i0 = b * IB + warp * 64 * P + 64 * q + lane, i1 = i0 + 32;
                if (!NB_IN(A.err, 53, i1 < A.npad)) i0 = i1 = 0;
                const float4 u = A.cp[i0 * kVmRecords], w = A.cp[i1 * kVmRecords];
                const float4 ug = A.cp[i0 * kVmRecords + 1], wg = A.cp[i1 * kVmRecords + 1];
                I.x[q] = make_float2(-u.x, -w.x);
                I.y[q] = make_float2(-u.y, -w.y);
                I.z[q] = make_float2(-u.z, -w.z);
                I.m[q] = make_float2(u.w, w.w);
                I.m3[q] = make_float2(3.f * u.w, 3.f * w.w);
                I.gx[q] = make_float2(ug.x, wg.x);
                I.gy[q] = make_float2(ug.y, wg.y);
                I.gz[q] = make_float2(ug.z, wg.z);
                I.gp[q] = make_float2(ug.w, wg.w);
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    ssum[(8 * q + r) * THREADS + tid] = zero2;
                    scmp[(8 * q + r) * THREADS + tid] = zero2;
                }
            }
        }

        const int s = k % STAGES;
        if (!mbar_wait_bounded(&full[s], (uint32_t)((k / STAGES) & 1), A.wait_ns)) {
            bad = 1;
            continue;
        }
        const float4 *tile = tiles + (size_t)s * JT * kVmRecords;
        put_at = (T.lin(b) - pj0 + t - b * TPB) * JT;
        float4 *dst = jsum + ((k & 1) * WARPS + warp) * 2 * JT + 2 * lane;
        // In the own block: the warp's own groups one-sided, others by met().
        const int64_t own = (t - b * TPB) * (JT / 32) - warp * 2 * P;
#pragma unroll 1
        for (int g = 0; g < JT / 32; ++g) {
            const float4 *G = tile + g * 32 * kVmRecords;
            float ja[kVmSums<GP>] = {};
            const int o = (int)own + g;
            if (t >= (b + 1) * TPB || met<WARPS, 2 * P>(o, warp, b & 1))
                vm_group<P, UNR, GP, true, RUN>(G, lane, -1, I, acc, ja, eps2);
            else if (o >= 0 && o < 2 * P)
                vm_group<P, 1, GP, false, 32>(G, lane, o, I, acc, ja, eps2);
            dst[64 * g] = make_float4(ja[0], ja[1], ja[2], ja[3]);
            if constexpr (GP) ja[7] = __fmaf_rn(3.f, ja[8], ja[7]);
            dst[64 * g + 1] = make_float4(ja[4], ja[5], ja[6], ja[7]);
            if (FOLD_IN_TILE && (g + 1) % FOLD == 0) fold();
        }
        if (!FOLD_IN_TILE && ++held == FOLD * 32 / JT) fold();
        if (++t == A.njt) {
            if (tid == 0) A.row_last[b] = (int)c;
            ++b;
            t = b * TPB;
        }
    }
    bad = __syncthreads_or(bad);
    if (!bad) {
        if (count > 0) put((count - 1) & 1);
        if (cur >= 0) flush(cur);
        return;
    }
    if (tid == 0) {
        atomicOr(A.err, kErrTimeout);
        // Let every copy still in flight land before this CTA's shared
        // memory is released.
        for (int s = 0; s < STAGES; ++s)
            if (issued_at[s] >= 0)
                mbar_wait_bounded(&full[s], (uint32_t)((issued_at[s] / STAGES) & 1), A.wait_ns);
    }
}

// As mutual_combine_kernel: 32 particles per block, their entries in contiguous
// shares for the warps, whose sums are added in warp order.
constexpr int kVmCombineWarps = 8;

__global__ void __launch_bounds__(32 * kVmCombineWarps) vjp_mutual_combine_kernel(const VmArgs A, const VmOut O) {
    __shared__ float part[kVmCombineWarps][16][32];
    pdl_wait_then_release();
    constexpr int K = 4;  // entries in flight
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = blockIdx.x * (int64_t)32 + lane;  // below the padded count
    const int ib = O.ib;
    const int64_t b = blockIdx.x * (int64_t)32 / ib, w = i - b * ib;
    float S[8] = {}, E[8] = {};
    const int64_t rend = b + 1 < A.r1 ? b + 1 : A.r1;
    const int rows = rend > A.r0 ? (int)(rend - A.r0) : 0;
    int c0 = 0, segs = 0;
    if (b >= A.r0 && b < A.r1) {  // (clamped: after a timeout the two words may be stale)
        c0 = max(A.row_first[b], 0);
        segs = max(min(A.row_last[b], A.grid - 1) - c0 + 1, 0);
    }
    const int e0 = (int)((int64_t)(rows + segs) * warp / kVmCombineWarps);
    const int e1 = (int)((int64_t)(rows + segs) * (warp + 1) / kVmCombineWarps);
    // Row r's entry of i is (lin(r) - lin(r0)) JT + i - r ib; the next row's is
    // (njt - r tpb) JT - ib further. R has the opposite sign there.
    const Triangle T{A.njt, A.nib, ib / O.jt};
    int64_t at = (T.lin(A.r0 + e0) - T.lin(A.r0)) * O.jt + i - (A.r0 + e0) * ib;
    int64_t step = (A.njt - (A.r0 + e0) * T.tpb) * O.jt - ib;
    for (int e = e0; e < e1 && e < rows; e += K) {
        float4 u[K], v[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            u[k] = v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (e + k < e1 && e + k < rows && NB_IN(A.err, 54, at >= 0 && 2 * at + 1 < A.pj_len)) {
                u[k] = __ldcg(A.pj + 2 * at);
                v[k] = __ldcg(A.pj + 2 * at + 1);
            }
            at += step;
            step -= ib;
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float h[8] = {-u[k].x, -u[k].y, -u[k].z, u[k].w, v[k].x, v[k].y, v[k].z, v[k].w};
            comp_add(S, E, h);
        }
    }
    for (int e = max(e0, rows); e < e1; ++e) {
        const int64_t o = (c0 + e - rows + b - A.r0) * 4 * (int64_t)ib + w;
        if (!NB_IN(A.err, 55, o >= 0 && o + 3 * ib < A.pi_len)) break;
        const float4 u = __ldcg(A.pi + o), v = __ldcg(A.pi + o + ib);
        const float4 ul = __ldcg(A.pi + o + 2 * ib), vl = __ldcg(A.pi + o + 3 * ib);
        const float h[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
        const float l[8] = {ul.x, ul.y, ul.z, ul.w, vl.x, vl.y, vl.z, vl.w};
        comp_add(S, E, h);
#pragma unroll
        for (int r = 0; r < 8; ++r) E[r] = __fsub_rn(E[r], l[r]);
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        part[warp][r][lane] = S[r];
        part[warp][8 + r][lane] = E[r];
    }
    __syncthreads();
    if (warp > 0 || i >= O.n) return;
#pragma unroll
    for (int r = 0; r < 8; ++r) S[r] = E[r] = 0.f;
    if (A.r0 > 0) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float4 s = O.state[4 * i + k], e = O.state[4 * i + 2 + k];
            S[4 * k] = s.x, S[4 * k + 1] = s.y, S[4 * k + 2] = s.z, S[4 * k + 3] = s.w;
            E[4 * k] = e.x, E[4 * k + 1] = e.y, E[4 * k + 2] = e.z, E[4 * k + 3] = e.w;
        }
    }
    for (int q = 0; q < kVmCombineWarps; ++q) {
        float h[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) h[r] = part[q][r][lane];
        comp_add(S, E, h);
#pragma unroll
        for (int r = 0; r < 8; ++r) E[r] = __fadd_rn(E[r], part[q][8 + r][lane]);
    }
    if (!O.last) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            O.state[4 * i + k] = make_float4(S[4 * k], S[4 * k + 1], S[4 * k + 2], S[4 * k + 3]);
            O.state[4 * i + 2 + k] = make_float4(E[4 * k], E[4 * k + 1], E[4 * k + 2], E[4 * k + 3]);
        }
        return;
    }
    const float4 u = A.cp[kVmRecords * i], g = A.cp[kVmRecords * i + 1];
    const float Sm = __fadd_rn(S[3], E[3]), gv[3] = {g.x, g.y, g.z};
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // gx = R + ga S - m V
        const float gx = __fmaf_rn(O.r_factor, __fadd_rn(S[c], E[c]),
                                   __fmaf_rn(-u.w, __fadd_rn(S[4 + c], E[4 + c]), __fmul_rn(gv[c], Sm)));
        if (!O.adj.lx) {
            O.gx[3 * i + c] = gx;
            continue;
        }
        const double x = O.adj.lx[3 * i + c] + (double)gx;
        O.adj.lx[3 * i + c] = x;
        double a = 0.0;
        if (!O.adj.first) {
            const double v = O.adj.lv[3 * i + c] + O.adj.dt * x;
            O.adj.lv[3 * i + c] = v;
            a = -((0.5 * O.adj.dt) * v);
        }
        O.adj.la[3 * i + c] = a;
    }
    const float gm = __fadd_rn(S[7], E[7]);
    if (O.adj.lx) O.adj.lm[i] = O.adj.lm[i] + (double)gm;
    else O.gm[i] = gm;
}

template <int WARPS, int P, int JT, int STAGES>
constexpr size_t vm_smem() {
    return (size_t)STAGES * JT * kVmRecords * sizeof(float4) + (size_t)4 * WARPS * JT * sizeof(float4) +
           (size_t)16 * P * WARPS * 32 * sizeof(float2) + (size_t)STAGES * (sizeof(uint64_t) + sizeof(int));
}

template <int W, int P, int J, int S, int U, int M, bool GP, int RUN, int FOLD>
static cudaError_t launch_vm(const VmArgs &a, size_t smem, cudaStream_t st) {
    return launch_with_pdl(vjp_mutual_kernel<W, P, J, S, U, M, GP, RUN, FOLD>, dim3((unsigned)a.grid), dim3(W * 32), smem,
                           st, a);
}

struct VmShape {
    int threads, ib, jt;
    const void *kernel;
    size_t smem;
    cudaError_t (*launch)(const VmArgs &, size_t, cudaStream_t);
};

#define NB_VM(J, U, GP, RUN, FOLD)                                                             \
    {128, 512, J, (const void *)vjp_mutual_kernel<4, 2, J, 3, U, 3, GP, RUN, FOLD>, vm_smem<4, 2, J, 3>(), \
     launch_vm<4, 2, J, 3, U, 3, GP, RUN, FOLD>}

// [size][without, with an upstream gradient on p]. Like the force's, register
// reads bound these: N = 65536 runs at 1332 G-pairs/s with gp and 1437 without it
// (direct kernels 1050 and 1175). Measured and not kept there: an unroll of 4
// (1228 / 1363) or 2 (1147 / 1283) with 128-particle tiles, four CTAs per SM (1159
// / 1256), 8 i-particles per thread at two CTAs (1277 / 1496, but 1043 / 1217
// against 1188 / 1333 at N = 16384).
// Runs. Without gp the direct kernels sum 64 or 128 l at a time and gm has nothing but
// sum s y^3 in it. With 128 terms to a run on both sides its error against FP64 was 1.04
// to 1.19 times theirs from N = 6000 to 16384; as below it is 0.83 to 0.96 (N = 8192
// 2.3e-7 -> 1.8e-7 and 60.9 -> 63.8 us, N = 16384 2.5e-7 -> 1.9e-7 and 197 -> 204 us;
// runs of 16 steps there 209 us). With gp 128 terms are no more than the direct
// kernel's.
static const VmShape kVmShapes[kVjpMutualSizes][2] = {
    {NB_VM(32, 4, false, 16, 2), NB_VM(32, 4, true, 32, 4)},
    {NB_VM(128, 8, false, 8, 2), NB_VM(128, 8, true, 32, 4)},
};
// The first without gp for the largest n, whose errors the longer runs do not raise
// above the direct kernels' (N = 20000 0.89 times, 298 us against 309).
static const VmShape kVmShapeLarge = NB_VM(32, 4, false, 32, 2);
#undef NB_VM
constexpr size_t kSmSharedBytes = 228 * 1024;

}  // namespace nbk

using namespace nbk;

namespace nbx {

nb_status run_vjp_mutual(nb_ctx *ctx, int size, const float *x, const float *m, int64_t n, float eps, const float *ga,
                         const float *gp, float *gx, float *gm, cudaStream_t st, const VjpState *state) {
    const VmShape &s = size == 0 && !gp && n >= kVjpMutualNoGpN ? kVmShapeLarge : kVmShapes[size][gp ? 1 : 0];
    PairVariant v{};
    v.tile.threads = s.threads;
    v.kernel = s.kernel;
    v.smem = s.smem;
    const int resident = resident_ctas(ctx, v, kSmSharedBytes / 2);
    const int64_t npad = round_up(std::max<int64_t>(n, 1), s.ib);
    const Triangle T{(n + s.jt - 1) / s.jt, (n + s.ib - 1) / s.ib, s.ib / s.jt};
    const int64_t most = (int64_t)(kMutualPartialBytes / (2 * sizeof(float4))) / s.jt;  // tiles per panel

    const TriangleScratch sizes = triangle_scratch(T, most);
    ExtState &es = ctx_ext(ctx);
    auto slot = [](MutualPart part) { return mutual_slot(kMutualVjp, part); };
    auto need = [&](MutualPart part, size_t bytes) {
        return ensure_buffer(&es.buf[slot(part)], &es.cap[slot(part)], bytes);
    };
    cudaError_t e = need(kPartCp, (size_t)npad * kVmRecords * sizeof(float4));
    if (e == cudaSuccess) e = need(kPartPi, (size_t)(resident + sizes.rows) * 4 * s.ib * sizeof(float4));
    if (e == cudaSuccess) e = need(kPartPj, (size_t)sizes.tiles * s.jt * 2 * sizeof(float4));
    if (e == cudaSuccess) e = need(kPartRows, (size_t)2 * T.nib * sizeof(int));
    if (e == cudaSuccess && sizes.panels) e = need(kPartState, (size_t)n * 4 * sizeof(float4));
    if (e != cudaSuccess) {
        if (e == cudaErrorMemoryAllocation) es.vjp_mutual_max_n = std::min(es.vjp_mutual_max_n, n - 1);
        return cuda_fail(ctx, e, "scratch allocation (mutual vjp)");
    }

    VmArgs A{};
    float4 *cp = static_cast<float4 *>(es.buf[slot(kPartCp)]);
    A.cp = cp;
    A.pi = static_cast<float4 *>(es.buf[slot(kPartPi)]);
    A.pj = static_cast<float4 *>(es.buf[slot(kPartPj)]);
    A.row_first = static_cast<int *>(es.buf[slot(kPartRows)]);
    A.row_last = A.row_first + T.nib;
    A.err = ctx_err_word(ctx);
    A.njt = T.njt;
    A.nib = T.nib;
    A.eps2 = eps * eps;
    A.fault_unit = ctx_fault_unit(ctx);
    A.wait_ns = ctx_wait_ns(ctx);
    A.npad = npad;
    A.pi_len = (int64_t)(es.cap[slot(kPartPi)] / sizeof(float4));
    A.pj_len = (int64_t)(es.cap[slot(kPartPj)] / sizeof(float4));
    VmOut O{gx,   gm,   state ? *state : VjpState{}, static_cast<float4 *>(es.buf[slot(kPartState)]), n, s.ib,
            s.jt, 0,    gp ? 3.f : 1.f};

    const dim3 pack((unsigned)((npad + 127) / 128));
    e = state ? launch_with_pdl(vjp_mutual_pack_state_kernel, pack, dim3(128), 0, st, *state, m, n, npad, cp)
              : launch_with_pdl(vjp_mutual_pack_kernel, pack, dim3(128), 0, st, x, m, ga, gp, n, npad, cp);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "vjp pack launch");
    for (int64_t r0 = 0; r0 < T.nib;) {
        const int64_t r1 = T.panel_end(r0, most);
        A.r0 = r0;
        A.r1 = r1;
        A.tiles = T.tiles(r0, r1);
        A.grid = triangle_grid(A.tiles, resident);
        // A grid that leaves places free asks for as much shared memory as keeps more
        // CTAs than needed off an SM: the places go to whichever SMs the pack has left,
        // and one with three CTAs takes as long as three (with gp, N = 4096, 288 CTAs for
        // 456 places: 33.3 us without, 27.1 with).
        const int sms = ctx_sm_count(ctx), per_sm = (A.grid + sms - 1) / sms;
        size_t smem = s.smem;
        if (per_sm * sms < resident) smem = std::max(smem, kSmSharedBytes / (per_sm + 1));
        {
            TimedLaunch t(ctx, 5, st);
            e = s.launch(A, smem, st);
        }
        if (e != cudaSuccess) return cuda_fail(ctx, e, "vjp kernel launch");
        O.last = r1 == T.nib;
        e = launch_with_pdl(vjp_mutual_combine_kernel, dim3((unsigned)((n + 31) / 32)), dim3(32 * kVmCombineWarps), 0,
                            st, A, O);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "vjp combine launch");
        r0 = r1;
    }
    return NB_OK;
}

}  // namespace nbx
