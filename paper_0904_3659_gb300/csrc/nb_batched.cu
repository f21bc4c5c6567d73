// nb_batched.cu -- Eq. (gravity) (Fujiwara & Nakasato, arXiv:0904.3659,
// Section "Introduction") for many independent clusters in one persistent
// launch, every unordered pair evaluated once, and the leap-frog of Section
// "Method" over such a batch (nb_batched.cuh has the layout and the work split).
//
// An evaluation is four launches: plan (padded offsets and blocks; a plan for the
// same sizes and offsets stands, and serves all steps of a call), pack (records and work items), pair kernel
// (its warps pop items from an atomic counter), combine. Every sum has a fixed
// order, so the results do not depend on which warp pops what.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>

#include "nb_batched.cuh"
#include "nb_device.cuh"
#include "nb_ext.h"
#include "nb_internal.h"
#include "nb_mutual.cuh"
#include "nb_triangle.cuh"

namespace nbk {
using namespace nbdev;

constexpr int kBmPlanThreads = 1024;
constexpr int kBmPlanNear = 8192;  // clusters whose first blocks the plan keeps in shared memory
// Items per SM that the plan aims at, 16 for a resident warp (12 on two-word records):
// more of them even out the end of the launch, fewer mean fewer partial sums. FP32
// records, 192 an SM against 144: 8 clusters of 6000 to 20000 540 us against 553, 500 of
// 4096 2868 against 2887 (one of 20000 206 against 164, where 144 happen to divide well);
// two-word records, 144 against 192: one of 20000 222 us a step against 261, the rest equal.
constexpr int64_t kItemsPerSm = 192, kItemsPerSmHL = 144;
constexpr int kBatchP = kBlock / 64;  // packed i-pairs per lane

struct BmBlock {  // a padded block
    int cluster, b, nt;  // block b of the cluster's nt
    int first;           // first item of its row
};

struct BmArgs {
    const int64_t *off;    // [C + 1] caller's offsets
    const float *eps;      // [C]
    int64_t C, n_total;
    int64_t cap_padded, cap_items;
    int64_t *poff;         // [C + 1] padded offsets
    int64_t *ibase;        // [C] the cluster's first item
    BmBlock *block;        // [cap_padded / kBlock]
    int4 *items;           // [cap_items] (cluster, i-block, first and end met tile)
    int *nitems, *head;    // item count and queue head
    BatchSplit *split;     // the batch's
    int64_t *pjbase;       // [C] the cluster's first j-side entry
    int64_t pj_entries;    // set aside
    int64_t want_items;    // items wanted (kItemsPerSm)
    int *notes;            // [C] what the pack found of a cluster (MutualNote); zero before it
    int *weights;          // [C] the form of its weights (MutualWeights), from the pair kernel
    MPart *cp;             // [cap_padded][1 or 2]
    float4 *pi;            // [item][kBlock] i-side sums
    float4 *pj;            // j-side sums (batch_pj_row)
    int *err;
    uint64_t wait_ns;
    // What the plan in the scratch was made for. fresh: nothing.
    BatchKey *planned;
    int64_t *planned_off;
    int fresh;
    int64_t pi_len, pj_len;
};

__host__ __device__ inline int64_t padded_size(int64_t n) {
    return n > 0 ? (n + kBlock - 1) / kBlock * kBlock : 0;
}

// Exclusive block-wide scan of one value per thread; *total the block's sum.
__device__ int64_t bm_scan(int64_t v, int64_t *total) {
    __shared__ int64_t wsum[kBmPlanThreads / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int64_t x = v;
    for (int d = 1; d < 32; d <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    __syncthreads();  // wsum of the scan before
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int64_t w = wsum[lane];
        for (int d = 1; d < 32; d <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += y;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    *total = wsum[kBmPlanThreads / 32 - 1];
    return x + (warp > 0 ? wsum[warp - 1] : 0) - v;
}

// Offsets and eps checked, padded offsets, every cluster's first item and every
// padded block's record (the items themselves are written by the pack's blocks).
// Offsets must start at 0, never decrease and end at n_total, and a non-empty
// cluster's eps must be > 0 with eps^2 a finite normal FP32 number; otherwise every
// cluster is given zero size, so that no kernel reads or writes. A plan for the same
// offsets stands (3 us; one is made in 25 us for 1024 clusters).
__global__ void __launch_bounds__(kBmPlanThreads) bm_plan_kernel(const BmArgs P) {
    pdl_wait_then_release();
    const int t = threadIdx.x;
    for (int64_t c = t; c < P.C; c += kBmPlanThreads) P.notes[c] = 0;
    if (t == 0) *P.head = 0;
    const BatchKey key{P.C, P.n_total, P.want_items, P.pj_entries};
    const int stands = !P.fresh && same_plan(*P.planned, key);
    int bad = 0, replan = !stands;
    for (int64_t c = t; c < P.C; c += kBmPlanThreads) {
        const int64_t o = P.off[c], end = P.off[c + 1];
        const float e = P.eps[c], e2 = e * e;
        if (stands) replan |= end != P.planned_off[c + 1];
        bad |= end < o;
        bad |= end > o && !(e > 0.f && e2 >= FLT_MIN && e2 <= FLT_MAX);  // also false for NaN
    }
    if (t == 0) bad |= (P.off[0] != 0) | (P.off[P.C] != P.n_total);
    if (!__syncthreads_or(bad | replan)) return;
    if (__syncthreads_or(bad)) {
        for (int64_t c = t; c <= P.C; c += kBmPlanThreads) P.poff[c] = 0;
        if (t == 0) {
            *P.nitems = 0;
            P.planned->clusters = -1;
            atomicOr(P.err, kErrBatchPlan);
        }
        return;
    }
    auto blocks = [&](int64_t c) { return c < P.C ? (int)(padded_size(P.off[c + 1] - P.off[c]) / kBlock) : 0; };
    __shared__ int longest;  // cluster, in blocks
    __shared__ int near[kBmPlanNear + 1];
    if (t == 0) longest = 1;
    int most = 1;
    int64_t carry = 0, met = 0, nit = 0, pj = 0, total;
    for (int64_t base = 0; base < P.C; base += kBmPlanThreads) {
        const int64_t c = base + t;
        const int nt = blocks(c);
        const int64_t ex = carry + bm_scan(nt, &total);
        if (c < P.C) P.poff[c] = ex * kBlock;
        if (c < kBmPlanNear) near[c] = (int)ex;
        carry += total;
        most = max(most, nt);
    }
    for (int d = 16; d > 0; d >>= 1) most = max(most, __shfl_xor_sync(0xffffffffu, most, d));
    if ((t & 31) == 0) atomicMax(&longest, most);
    __syncthreads();
    // The longest band whose j-side sums fit: that of the longest cluster, or by bisection.
    auto need = [&](int band) {
        int64_t mine = 0, all;
        for (int64_t c = t; c < P.C; c += kBmPlanThreads) mine += batch_pj_need(band, blocks(c));
        bm_scan(mine, &all);
        return all;
    };
    int band = longest;
    if (need(band) > P.pj_entries) {
        int lo = 1;  // (needs nothing)
        while (band - lo > 1) {
            const int mid = (lo + band) / 2;
            if (need(mid) <= P.pj_entries) lo = mid;
            else band = mid;
        }
        band = lo;
    }
    for (int64_t base = 0; base < P.C; base += kBmPlanThreads) {
        bm_scan(batch_met(band, blocks(base + t)), &total);
        met += total;
    }
    const BatchSplit split = batch_split(band, longest, met, P.want_items);
    if (t == 0) {
        P.poff[P.C] = carry * kBlock;
        *P.split = split;
    }
    for (int64_t base = 0; base < P.C; base += kBmPlanThreads) {
        const int64_t c = base + t;
        const int nt = blocks(c);
        const int64_t ex = bm_scan(nt > 0 ? split.first(nt, nt) : 0, &total);
        if (c < P.C) P.ibase[c] = nit + ex;
        nit += total;
        const int64_t px = bm_scan(batch_pj_need(band, nt), &total);
        if (c < P.C) P.pjbase[c] = pj + px;
        pj += total;
    }
    const bool ok = carry * kBlock <= P.cap_padded && nit <= P.cap_items;
    __syncthreads();  // poff, ibase, near
    // Each padded block's cluster: the last one that starts at or before it.
    for (int64_t s = t; ok && s < carry; s += kBmPlanThreads) {
        int64_t lo = 0, hi = P.C;
        while (hi - lo > 1) {
            const int64_t mid = (lo + hi) / 2;
            const int64_t at = P.C <= kBmPlanNear ? near[mid] : P.poff[mid] / kBlock;
            if (at <= s) lo = mid;
            else hi = mid;
        }
        const int64_t b0 = P.C <= kBmPlanNear ? near[lo] : P.poff[lo] / kBlock;
        const int nt = blocks(lo), b = (int)(s - b0);
        P.block[s] = BmBlock{(int)lo, b, nt, (int)(P.ibase[lo] + split.first(nt, b))};
    }
    __syncthreads();  // poff is read above
    if (t == 0) {
        *P.nitems = ok ? (int)nit : 0;
        if (!ok) atomicOr(P.err, kErrBatchPlan);
        *P.planned = key;
        if (!ok) P.planned->clusters = -1;
    }
    for (int64_t c = t; c <= P.C; c += kBmPlanThreads) {
        if (!ok) P.poff[c] = 0;
        P.planned_off[c] = P.off[c];
    }
}

// One block of the pack: record r (and lo) of the block's particle, its notes,
// and the items of the block's row.
template <bool HL>
__device__ __forceinline__ void bm_put(const BmArgs &A, const BmBlock &B, bool real, const MPart &r, const MPart &lo,
                                       float hm0) {
    const int t = threadIdx.x, c = B.cluster;
    const BatchSplit split = *A.split;
    const float eps = A.eps[c];
    if (!(eps >= 1.f / kMutualRange && eps <= kMutualRange) && t == 0) atomicOr(&A.notes[c], (int)kNoteWide);
    mutual_note(real, r, hm0, eps, &A.notes[c]);
    MPart *dst = A.cp + ((int64_t)blockIdx.x * kBlock + t) * (HL ? kHLRecords : 1);
    dst[0] = r;
    if (HL) dst[1] = lo;
    const int met = B.nt - B.b % cluster_band(split.band, B.nt), q = split.items(met);
    for (int k = t; k < q; k += kBlock) {
        int v0, v1;
        split.range(B.nt, met, k, &v0, &v1);
        if (NB_IN(A.err, 60, (int64_t)B.first + k < A.cap_items)) A.items[B.first + k] = make_int4(c, B.b, v0, v1);
    }
}

// Pack padded rows from FP32 or FP64 positions (rounded to FP32). KICK: the kicks
// (kick_back: the previous step's too) and the drift of the leap-frog first.
template <typename T, bool KICK>
__global__ void __launch_bounds__(kBlock) bm_pack_kernel(const BmArgs A, T *__restrict__ x, double *__restrict__ v,
                                                         const float *__restrict__ a, const float *__restrict__ m,
                                                         double dt, int kick_back) {
    pdl_wait();
    if ((int64_t)blockIdx.x * kBlock >= A.poff[A.C]) return;
    const BmBlock B = A.block[blockIdx.x];
    const int64_t c = B.cluster, li = (int64_t)B.b * kBlock + threadIdx.x, o = A.off[c], nc = A.off[c + 1] - o;
    MPart r = mutual_padding();
    if (li < nc) {
        const int64_t i = o + li;
        float q[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int64_t e = 3 * i + k;
            T xc = x[e];
            if constexpr (KICK) {
                const double h = 0.5 * dt, g = -(double)a[e];
                double vc = v[e];
                if (kick_back) vc = vc + h * g;  // Eq. (3) of the previous step
                vc = vc + h * g;                 // Eq. (1)
                xc = xc + dt * vc;               // Eq. (2)
                v[e] = vc;
                x[e] = xc;
            }
            q[k] = (float)xc;
        }
        r = make_float4(-q[0], -q[1], -q[2], -0.5f * m[i]);
    }
    bm_put<false>(A, B, li < nc, r, r, -0.5f * m[o]);
}

// Order-preserving map of an FP64 value's bits to a signed 64-bit integer
// (its own inverse): the bounding box below is reduced with integer min/max,
// which run at the integer pipe's rate rather than the FP64 pipe's.
__device__ __forceinline__ long long ordered_key(long long bits) {
    return bits >= 0 ? bits : bits ^ 0x7fffffffffffffffll;
}

constexpr int kFrameThreads = 512;

// Compensated mode on FP64 state, first pass: the frame of cluster
// blockIdx.x, the centre of its bounding box and the grid 2^(E-23) set by
// the box's half-width (all pairs lie inside one cluster, so each cluster
// has its own frame): frame[c] = (centre, grid). Positions are finite.
__global__ void __launch_bounds__(kFrameThreads) batch_frame_kernel(const double *__restrict__ x,
                                                                    const int64_t *__restrict__ off,
                                                                    const int64_t *__restrict__ poff,
                                                                    double4 *__restrict__ frame) {
    __shared__ long long s[6][kFrameThreads / 32];
    pdl_wait();
    const int64_t c = blockIdx.x;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t o = off[c], psz = poff[c + 1] - poff[c];
    const int64_t nc = psz > 0 ? off[c + 1] - o : 0;
    if (psz <= 0) return;
    const long long *xb = reinterpret_cast<const long long *>(x) + 3 * o;
    long long lo[3] = {LLONG_MAX, LLONG_MAX, LLONG_MAX}, hi[3] = {LLONG_MIN, LLONG_MIN, LLONG_MIN};
#pragma unroll 4
    for (int64_t li = t; li < nc; li += kFrameThreads)
        for (int k = 0; k < 3; ++k) {
            const long long v = ordered_key(xb[3 * li + k]);
            lo[k] = v < lo[k] ? v : lo[k];
            hi[k] = v > hi[k] ? v : hi[k];
        }
    for (int k = 0; k < 3; ++k)
        for (int d = 16; d > 0; d >>= 1) {
            const long long a = __shfl_xor_sync(0xffffffffu, lo[k], d);
            const long long b = __shfl_xor_sync(0xffffffffu, hi[k], d);
            lo[k] = a < lo[k] ? a : lo[k];
            hi[k] = b > hi[k] ? b : hi[k];
        }
    if (lane == 0)
        for (int k = 0; k < 3; ++k) {
            s[k][warp] = lo[k];
            s[3 + k][warp] = hi[k];
        }
    __syncthreads();
    if (t == 0) {
        double cen[3], ext = 0.0;
        for (int k = 0; k < 3; ++k) {
            long long l = s[k][0], h = s[3 + k][0];
            for (int w = 1; w < kFrameThreads / 32; ++w) {
                l = s[k][w] < l ? s[k][w] : l;
                h = s[3 + k][w] > h ? s[3 + k][w] : h;
            }
            const double dl = __longlong_as_double(ordered_key(l)), dh = __longlong_as_double(ordered_key(h));
            cen[k] = 0.5 * (dl + dh);
            ext = fmax(ext, 0.5 * (dh - dl));
        }
        frame[c] = make_double4(cen[0], cen[1], cen[2], ldexp(1.0, hl_grid_exponent(ext) - 23));
    }
}

// Compensated mode on FP64 state: HL records in the cluster's frame (centre of
// its bounding box, grid; see kHLRecords).
__global__ void __launch_bounds__(kBlock) bm_pack_hl_kernel(const BmArgs A, const double *__restrict__ x,
                                                            const float *__restrict__ m,
                                                            const double4 *__restrict__ frame) {
    pdl_wait();
    if ((int64_t)blockIdx.x * kBlock >= A.poff[A.C]) return;
    const BmBlock B = A.block[blockIdx.x];
    const int64_t c = B.cluster, li = (int64_t)B.b * kBlock + threadIdx.x, o = A.off[c], nc = A.off[c + 1] - o;
    MPart hi = mutual_padding(), lo = make_float4(0.f, 0.f, 0.f, 0.f);
    if (li < nc) {
        const double4 f = frame[c];
        const double cen[3] = {f.x, f.y, f.z};
        const double magic = 6755399441055744.0 * f.w;  // 1.5 * 2^52 * grid
        const int64_t i = o + li;
        float h[3], l[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double y = __dsub_rn(x[3 * i + k], cen[k]);
            const double yh = __dsub_rn(__dadd_rn(y, magic), magic);
            h[k] = (float)yh;
            l[k] = (float)__dsub_rn(y, yh);
        }
        hi = make_float4(-h[0], -h[1], -h[2], -0.5f * m[i]);
        lo = make_float4(-l[0], -l[1], -l[2], 0.f);
    }
    bm_put<true>(A, B, li < nc, hi, lo, -0.5f * m[o]);
}

// The sums of a cluster of kDirectBlocks blocks or fewer are those of one evaluation
// per (i, j): the masses in the weights, a block's j in order in one FP32 sum of 128
// terms, the blocks' sums compensated. Their particles are the heaviest of a batch of
// clusters of equal mass and their accelerations the least averaged.
__device__ __forceinline__ int cluster_weights(const BmArgs &A, int c, int nt) {
    return nt <= kDirectBlocks ? kWide : mutual_weights(__ldcg(A.notes + c));
}

// A group's particles on the first Q pairs of i-slots, for the i-side only; the
// particles of slot `self` (-1: none) do not meet themselves. w = (f y) y^2 with f = 1
// where all masses are equal, c m_i m_j (PRODUCT) or m_j. On FP32 records a loop of its
// own for PRODUCT and packed differences, the broadcast j costing a move per value: 2300
// clusters of 200 particles 124 -> 112 us a call, 1900 of 256 108 -> 100, 1024 up to 512
// 60 -> 53. Two-word records take one loop for both, the kernel's loops then staying in
// the instruction cache (1024 up to 512, unequal masses: 91 us a step, 102 with two),
// and scalar differences (packed 1 to 2% slower), but a short loop of its own, without
// the test for the own particle, for other blocks where no product is formed (2500
// clusters of 200 a step 201 -> 195 us, 1900 of 256 178 -> 175).
template <int P, int Q, bool HL, bool PRODUCT, bool SELF = true>
__device__ __forceinline__ void one_sided_loop(int weights, const MPart *__restrict__ T, int lane, int self,
                                               const MutualI<P, HL> &I, float2 (&acc)[P][4], const float2 eps2) {
    const bool equal = weights == kEqual, product = PRODUCT && (!HL || weights == kProduct);
#pragma unroll (SELF ? 4 : 2)
    for (int t = 0; t < 32; ++t) {
        const float4 h = T[HL ? 2 * t : t];
        const float4 l = HL ? T[2 * t + 1] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float hj = equal ? 1.f : h.w;
        const int own = SELF && t == lane ? self : -1;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            float2 dx, dy, dz;
            if constexpr (HL) {
                mutual_diff<P, HL>(I, q, h, l, dx, dy, dz);
            } else {
                dx = add2(I.x[q], splat2(h.x));
                dy = add2(I.y[q], splat2(h.y));
                dz = add2(I.z[q], splat2(h.z));
            }
            float2 s = fma2(dx, dx, eps2);
            s = fma2(dy, dy, s);
            s = fma2(dz, dz, s);
            const float2 y = make_float2(rsqrt_sfu(s.x), rsqrt_sfu(s.y));
            float2 f = splat2(hj);  // (left out here: an infinite mass times y = 0 would be NaN)
            if (SELF && own == 2 * q) f.x = 0.f;
            if (SELF && own == 2 * q + 1) f.y = 0.f;
            if (product) f = make_float2(__fmul_rn(I.hm[q].x, f.x), __fmul_rn(I.hm[q].y, f.y));
            const float2 p = mul2(f, y);
            acc[q][3] = add2(acc[q][3], p);
            const float2 w = mul2(p, mul2(y, y));
            acc[q][0] = fma2(w, dx, acc[q][0]);
            acc[q][1] = fma2(w, dy, acc[q][1]);
            acc[q][2] = fma2(w, dz, acc[q][2]);
        }
    }
}

template <int P, int Q, bool HL>
__device__ __forceinline__ void one_sided_group(int weights, const MPart *__restrict__ T, int lane, int self,
                                                const MutualI<P, HL> &I, float2 (&acc)[P][4], const float2 eps2) {
    if (HL && self < 0 && weights != kProduct)
        one_sided_loop<P, Q, HL, false, false>(weights, T, lane, self, I, acc, eps2);
    else if (HL || weights == kProduct) one_sided_loop<P, Q, HL, true>(weights, T, lane, self, I, acc, eps2);
    else one_sided_loop<P, Q, HL, false>(weights, T, lane, self, I, acc, eps2);
}

struct BmStage {
    int item, cluster, iblock, tile, end;
    int len;  // particles copied into the stage
    int last;  // no particles of the cluster follow
};

// One warp per CTA, persistent: lane 0 pops items and issues the 1-D bulk copies
// of the tiles they meet, the warp consumes them. Later blocks of the band are met
// as in mutual_kernel (nb_mutual.cu), each pair for both sides, the rest with
// one_sided_group: in a row's own block both orders of a pair cost 24 operations
// against 18 and the moves, but no chain through the lanes and no code of its own
// (the mutual form there, with a loop for each slot, measured 62 against 57 us on
// 1024 clusters of up to 512 particles, 663 against 667 us up to 4096).
//
// Bound by the register-file reads of the pair loop, and for small clusters by the
// items' ends. 128 particles a block (4 per lane) against 256: half the padding and
// half the own-block work, twice the j-side sums; 57 against 87 us up to 512, 667
// against 687 up to 4096. Tiles of 64 against 128: 47 against 55 us up to 512.
// Twelve warps an SM (140 registers a lane, 147 on two-word records).
// Against one evaluation per (i, j): 1024 clusters up to 4096 particles 817 -> 685 us
// (the pair kernel 777 -> 632; 904.8e6 unordered pairs, 66% of the FP32 lanes' issue
// rate counting 18 operations a pair and the padding), 1024 up to 512 82 -> 53, 300
// up to 2048 113 -> 81, a step of those on FP64 state 150 -> 116.
template <int STAGES, int MINB, int UNR, bool HL>
__global__ void __launch_bounds__(32, MINB) bm_pair_kernel(const BmArgs A) {
    constexpr int P = kBatchP;
    constexpr int RS = HL ? kHLRecords : 1;
    constexpr uint32_t TILE_BYTES = kTile * RS * sizeof(MPart);

    // Shared memory: [STAGES tiles][running sums, carries][barriers][stages][issue records]
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x;
    MPart *tiles = reinterpret_cast<MPart *>(smem);
    float2 *ssum = reinterpret_cast<float2 *>(smem + (size_t)STAGES * TILE_BYTES);
    float2 *scmp = ssum + 4 * P * 32;
    uint64_t *full = reinterpret_cast<uint64_t *>(scmp + 4 * P * 32);
    BmStage *meta = reinterpret_cast<BmStage *>(full + STAGES);
    int *issued_at = reinterpret_cast<int *>(meta + STAGES);

    if (lane == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            issued_at[s] = -1;
        }
        fence_mbar_init();
    }
    __syncwarp();
    // (No release: the combine's blocks, resident early, slow small batches: 40 clusters
    // up to 1024 27.6 -> 23.5 us, 32 compensated steps of 40 up to 512 1022 -> 919.)
    pdl_wait();

    // Producer state (lane 0): walks the (item, tile) stream.
    int p_item = -1, p_cluster = 0, p_b = 0, p_nt = 0, p_v = 0, p_end = 0, p_done = 0;
    int64_t p_row0 = 0, p_nc = 0;
    const int nitems = *A.nitems, band = A.split->band;
    auto produce = [&](int kk) {
        const int s = kk % STAGES;
        BmStage mt;
        int tile = 0;
        for (;;) {  // the next tile that holds particles
            if (p_v < p_end) {
                tile = batch_met_tile(band, p_nt, p_b, p_v++);
                if ((int64_t)tile * kTile < p_nc) break;
                continue;
            }
            const int it = p_done ? nitems : atomicAdd(A.head, 1);
            if (it >= nitems || !NB_IN(A.err, 61, it < A.cap_items)) {
                p_done = 1;
                break;
            }
            const int4 w = A.items[it];
            p_item = it;
            p_cluster = w.x;
            p_b = w.y;
            p_v = w.z;
            p_end = w.w;
            p_row0 = A.poff[w.x];
            p_nt = (int)((A.poff[w.x + 1] - p_row0) / kBlock);
            p_nc = A.off[w.x + 1] - A.off[w.x];
        }
        if (!p_done && !NB_IN(A.err, 62, p_row0 + (int64_t)(tile + 1) * kTile <= A.cap_padded)) p_done = 1;
        mt.item = p_item;
        mt.cluster = p_cluster;
        mt.iblock = p_b;
        mt.tile = tile;
        // The cluster's last tile stops at its last particle, rounded up to 32.
        const int64_t rem = p_nc - (int64_t)tile * kTile;
        mt.len = rem >= kTile ? kTile : (int)((rem + 31) & ~(int64_t)31);
        mt.last = rem <= kTile;
        mt.end = p_done;
        meta[s] = mt;
        if (p_done) {
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&full[s])) : "memory");
        } else {
            issued_at[s] = kk;
            const uint32_t bytes = (uint32_t)mt.len * RS * (uint32_t)sizeof(MPart);
            mbar_arrive_expect_tx(&full[s], bytes);
            bulk_g2s(tiles + (size_t)s * kTile * RS, A.cp + (p_row0 + (int64_t)tile * kTile) * RS, bytes, &full[s]);
        }
    };
    if (lane == 0)
        for (int kk = 0; kk < STAGES - 1; ++kk) produce(kk);

    const float2 zero2 = splat2(0.f);
    MutualI<P, HL> I;
    float2 acc[P][4];
#pragma unroll
    for (int q = 0; q < P; ++q)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[q][r] = zero2;
    int cur_item = -1, weights = kEqual, b = 0, slots = 0, band_end = 0;
    bool direct = false;
    float4 *pj = nullptr;  // the row's j-side entries, from its block b + 1 on
    float2 eps2 = zero2;

    // Kahan: the true value is sum - carry. After every tile: the error against FP64
    // stays below that of one evaluation per (i, j) (9.0e-8 against 1.01e-7 up to 4096
    // particles a cluster; every 256 particles 9.9e-8 and no faster).
    auto fold = [&]() {
#pragma unroll
        for (int q = 0; q < P; ++q)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int k = (4 * q + r) * 32 + lane;
                const float2 s0 = ssum[k];
                const float2 y = add2(acc[q][r], neg2(scmp[k]));
                const float2 v = add2(s0, y);
                scmp[k] = add2(add2(v, neg2(s0)), neg2(y));
                ssum[k] = v;
                acc[q][r] = zero2;
            }
    };
    auto write_out = [&]() {
        if (!NB_IN(A.err, 63, ((int64_t)cur_item + 1) * kBlock <= A.pi_len)) return;
        float4 *dst = A.pi + (int64_t)cur_item * kBlock + lane;
#pragma unroll
        for (int q = 0; q < P; ++q) {
            float2 s[4];
#pragma unroll
            for (int r = 0; r < 4; ++r)
                s[r] = add2(ssum[(4 * q + r) * 32 + lane], neg2(scmp[(4 * q + r) * 32 + lane]));
            dst[64 * q] = make_float4(s[0].x, s[1].x, s[2].x, s[3].x);
            dst[64 * q + 32] = make_float4(s[0].y, s[1].y, s[2].y, s[3].y);
        }
    };

    int bad = 0;
    for (int k = 0;; ++k) {
        // All lanes are done with iteration k-1: its stage may be refilled.
        __syncwarp();
        if (lane == 0) produce(k + STAGES - 1);
        const int s = k % STAGES;
        if (!mbar_wait_bounded(&full[s], (uint32_t)((k / STAGES) & 1), A.wait_ns)) bad = 1;
        if (__any_sync(0xffffffffu, bad)) {
            bad = 1;
            break;
        }
        const BmStage mt = meta[s];
        if (mt.end) break;
        if (mt.item != cur_item) {
            if (cur_item >= 0) write_out();
            cur_item = mt.item;
            b = mt.iblock;
            const float eps = A.eps[mt.cluster];
            eps2 = splat2(eps * eps);
            const int64_t row0 = A.poff[mt.cluster], nc = A.off[mt.cluster + 1] - A.off[mt.cluster];
            const int nt = (int)((A.poff[mt.cluster + 1] - row0) / kBlock), cb = cluster_band(band, nt), s0 = b / cb * cb;
            weights = cluster_weights(A, mt.cluster, nt);
            if (lane == 0 && b == 0) A.weights[mt.cluster] = weights;
            direct = nt <= kDirectBlocks;
            band_end = min(s0 + cb, nt);
            slots = (int)min((nc - (int64_t)b * kBlock + 31) / 32, (int64_t)(2 * P));
            pj = A.pj + A.pjbase[mt.cluster] + batch_pj_row(band, nt, b);
            const float hm0 = A.cp[row0 * RS].w;
#pragma unroll
            for (int q = 0; q < P; ++q) {
                int64_t i0 = row0 + (int64_t)b * kBlock + 64 * q + lane, i1 = i0 + 32;
                if (!NB_IN(A.err, 64, i1 < A.cap_padded)) i0 = i1 = 0;
                const float4 u = A.cp[i0 * RS], w = A.cp[i1 * RS];
                I.x[q] = make_float2(-u.x, -w.x);
                I.y[q] = make_float2(-u.y, -w.y);
                I.z[q] = make_float2(-u.z, -w.z);
                I.hm[q] = make_float2(u.w, w.w);
                if (weights == kProduct)
                    I.hm[q] = make_float2(mutual_scale(u.w, hm0, eps), mutual_scale(w.w, hm0, eps));
                if constexpr (HL) {
                    const float4 ul = A.cp[i0 * RS + 1], wl = A.cp[i1 * RS + 1];
                    I.lx[q] = make_float2(-ul.x, -wl.x);
                    I.ly[q] = make_float2(-ul.y, -wl.y);
                    I.lz[q] = make_float2(-ul.z, -wl.z);
                }
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    ssum[(4 * q + r) * 32 + lane] = scmp[(4 * q + r) * 32 + lane] = zero2;
            }
        }
        const MPart *T = tiles + (size_t)s * kTile * RS;
        const int groups = mt.len / 32, block = mt.tile / kBlockTiles;
        if (block > b && block < band_end) {
            float4 *dst = pj + ((int64_t)mt.tile * kTile - (int64_t)(b + 1) * kBlock) + lane;
            if (NB_IN(A.err, 65, dst >= A.pj && dst + kTile - lane <= A.pj + A.pj_len))
#pragma unroll 1
                for (int g = 0; g < groups; ++g) {
                    float ja[4];
                    run_group<P, UNR, true, HL, kAny>(weights, T + g * 32 * RS, lane, I, acc, ja, eps2);
                    dst[32 * g] = make_float4(ja[0], ja[1], ja[2], ja[3]);
                }
        } else {
            const int g0 = block == b ? mt.tile % kBlockTiles * (kTile / 32) : -kTile;
#pragma unroll 1
            for (int g = 0; g < groups; ++g) {
                const MPart *G = T + g * 32 * RS;
                const int self = g0 < 0 ? -1 : g0 + g;
                if (slots > 2) one_sided_group<P, P, HL>(weights, G, lane, self, I, acc, eps2);
                else one_sided_group<P, 1, HL>(weights, G, lane, self, I, acc, eps2);
            }
        }
        if (!direct || mt.last || mt.tile % kBlockTiles == kBlockTiles - 1) fold();
    }
    if (!bad) {
        if (cur_item >= 0) write_out();
        return;
    }
    if (lane == 0) {
        atomicOr(A.err, kErrTimeout);
        // Let this warp's copies in flight land before the CTA can exit.
        for (int s = 0; s < STAGES; ++s)
            if (issued_at[s] >= 0)
                mbar_wait_bounded(&full[s], (uint32_t)((issued_at[s] / STAGES) & 1), A.wait_ns);
    }
    __syncwarp();
}

// Per particle: the j-side sums of the earlier rows of its band, in row order, then
// the items of its own row, in chunk order; then the factors the weights left out.
template <bool HL>
__global__ void __launch_bounds__(kBlock) bm_combine_kernel(const BmArgs A, float *__restrict__ a,
                                                            float *__restrict__ p) {
    pdl_wait_then_release();
    constexpr int RS = HL ? kHLRecords : 1;
    if ((int64_t)blockIdx.x * kBlock >= A.poff[A.C]) return;  // (zero when the plan rejected the offsets)
    const BmBlock B = A.block[blockIdx.x];
    const BatchSplit split = *A.split;
    const int c = B.cluster, b = B.b, nt = B.nt;
    const int64_t row0 = (int64_t)(blockIdx.x - b) * kBlock;
    const int64_t li = (int64_t)b * kBlock + threadIdx.x, o = A.off[c], nc = A.off[c + 1] - o;
    // For the next evaluation of the call, which has no plan before it.
    if (threadIdx.x == 0 && b == 0) A.notes[c] = 0;
    if (threadIdx.x == 0 && blockIdx.x == 0) *A.head = 0;
    if (li >= nc) return;
    float S[4] = {0.f, 0.f, 0.f, 0.f}, E[4] = {0.f, 0.f, 0.f, 0.f};
    constexpr int K = 8;  // loads in flight
    const int cb = cluster_band(split.band, nt), s0 = b / cb * cb, len = min(s0 + cb, nt) - s0;
    const int64_t pj0 = A.pjbase[c] + batch_pj_row(split.band, nt, s0) + threadIdx.x;
    for (int r = s0; r < b; r += K) {
        float4 v[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r + k >= b) continue;
            const int64_t e = r + k - s0;  // rows before it in the band
            const int64_t at = pj0 + (e * len - e * (e + 1) / 2 + (b - r - k - 1)) * kBlock;
            if (NB_IN(A.err, 66, at < A.pj_len)) v[k] = __ldcg(A.pj + at);
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (r + k >= b) break;
            const float h[4] = {-v[k].x, -v[k].y, -v[k].z, v[k].w};
            comp_add(S, E, h);
        }
    }
    const int met = nt - (b - s0), q = split.items(met);
    for (int j = 0; j < q; j += K) {
        float4 u[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            u[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j + k >= q) continue;
            if (split.parts > 1) {  // a part past the last particle was not evaluated
                int v0, v1;
                split.range(nt, met, j + k, &v0, &v1);
                if (v0 == v1 || (int64_t)batch_met_tile(split.band, nt, b, v0) * kTile >= nc) continue;
            }
            const int64_t at = ((int64_t)B.first + j + k) * kBlock + threadIdx.x;
            if (NB_IN(A.err, 67, at < A.pi_len)) u[k] = __ldcg(A.pi + at);
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (j + k >= q) break;
            const float h[4] = {u[k].x, u[k].y, u[k].z, u[k].w};
            comp_add(S, E, h);
        }
    }
    const float hm0 = A.cp[row0 * RS].w;
    const int weights = __ldcg(A.weights + c);
    const float hm = A.cp[((int64_t)blockIdx.x * kBlock + threadIdx.x) * RS].w;
    const float f = weights == kProduct ? mutual_scale(hm, hm0, A.eps[c]) : hm0;
    float v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) v[r] = mutual_result(weights, S[r], E[r], f);
    const int64_t i = o + li;
    if (!NB_IN(A.err, 68, i >= 0 && i < A.n_total)) return;
    a[3 * i + 0] = v[0];
    a[3 * i + 1] = v[1];
    a[3 * i + 2] = v[2];
    p[i] = v[3];
}

template <int S, bool HL>
constexpr size_t bm_smem() {
    return (size_t)S * (kTile * (HL ? kHLRecords : 1) * sizeof(MPart) + sizeof(uint64_t) + sizeof(BmStage) +
                        sizeof(int)) + (size_t)2 * 4 * kBatchP * 32 * sizeof(float2);
}

// Leap-frog pieces that do not pack (the batched pack follows them).
__global__ void batch_kick_drift_kernel(double *__restrict__ x, double *__restrict__ v,
                                        const float *__restrict__ a, int64_t n, double dt,
                                        int kick_back) {
    pdl_wait_then_release();
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= 3 * n) return;
    const double h = 0.5 * dt, g = -(double)a[k];
    double vc = v[k];
    if (kick_back) vc = vc + h * g;  // Eq. (3) of the previous step
    vc = vc + h * g;                 // Eq. (1)
    v[k] = vc;
    x[k] = x[k] + dt * vc;           // Eq. (2)
}

__global__ void batch_kick_kernel(double *__restrict__ v, const float *__restrict__ a, int64_t n,
                                  double dt) {
    pdl_wait_then_release();
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= 3 * n) return;
    v[k] = v[k] + (0.5 * dt) * (-(double)a[k]);  // Eq. (3)
}

}  // namespace nbk

using namespace nbk;
using namespace nbx;

namespace {

constexpr int kBmStages = 3;
constexpr auto kBmPair = bm_pair_kernel<kBmStages, 12, 4, false>;
constexpr auto kBmPairHL = bm_pair_kernel<kBmStages, 12, 4, true>;
// Of a tiny cluster's item little is arithmetic: more warps (16 an SM, 128 registers a
// lane) hide more of the rest. 100000 clusters of 8 particles 510 -> 473 us, of 64 703 ->
// 671; the same at 100, 128 particles 67 -> 73 us.
constexpr auto kBmPairTiny = bm_pair_kernel<kBmStages, 16, 4, false>;
constexpr int64_t kTinyMean = 64;  // particles per cluster

struct BatchCall {
    const int64_t *offsets;
    int64_t C, n_total;
    const float *eps;
    bool hl;  // HL records (compensated mode on FP64 state)
};

auto bm_kernel(const BatchCall &k) { return k.hl ? kBmPairHL : k.n_total <= kTinyMean * k.C ? kBmPairTiny : kBmPair; }

PairVariant bm_variant(const BatchCall &k) {
    PairVariant v{};
    v.tile.threads = 32;
    v.kernel = (const void *)bm_kernel(k);
    v.smem = k.hl ? bm_smem<kBmStages, true>() : bm_smem<kBmStages, false>();
    return v;
}

// Where a call's positions come from: FP32, or FP64 state with the leap-frog's
// kicks and drift to be applied first (kick).
struct BatchSource {
    const float *x32;
    double *x64, *v;
    const float *a, *m;
    double dt;
    int kick, kick_back;
};

nb_status bm_args(nb_ctx *ctx, const BatchCall &k, bool small, BmArgs *out) {
    ExtState &es = ctx_ext(ctx);
    BmArgs A{};
    A.off = k.offsets;
    A.eps = k.eps;
    A.C = k.C;
    A.n_total = k.n_total;
    A.cap_padded = k.n_total + k.C * (int64_t)kBlock;
    const int64_t blocks = A.cap_padded / kBlock;
    // small: one item per row and no j-side sums.
    A.want_items = small ? 1 : (k.hl ? kItemsPerSmHL : kItemsPerSm) * ctx_sm_count(ctx);
    A.cap_items = blocks + A.want_items + 1;  // at most one per row beyond the number wanted
    if (A.cap_items > INT_MAX || k.C > INT_MAX) return fail(ctx, NB_ERR_ARG, "batch too large for 32-bit work items");
    A.pj_entries = small ? 0 : batch_pj_entries(k.C, k.n_total);
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    // [the plan's key, item count, queue head, split][poff][ibase][pjbase][planned offsets][notes][weights][padded blocks]
    const size_t b_off = al((size_t)(k.C + 1) * sizeof(int64_t)), b_c = al((size_t)k.C * sizeof(int));
    const size_t b_blk = al((size_t)blocks * sizeof(BmBlock));
    const size_t plan_before = es.cap[SLOT_BATCH_PLAN];
    cudaError_t e = cudaSuccess;
    auto need = [&](int slot, size_t bytes) {
        if (e == cudaSuccess) e = ensure_buffer(&es.buf[slot], &es.cap[slot], bytes);
    };
    need(SLOT_BATCH_PLAN, 256 + 4 * b_off + 2 * b_c + b_blk);
    if (es.cap[SLOT_BATCH_PLAN] != plan_before) es.batch_plan = false;
    need(SLOT_BATCH_ITEMS, (size_t)A.cap_items * sizeof(int4));
    need(SLOT_BATCH_CP, (size_t)A.cap_padded * (k.hl ? kHLRecords : 1) * sizeof(MPart));
    need(SLOT_BATCH_PI, (size_t)A.cap_items * kBlock * sizeof(float4));
    need(SLOT_BATCH_PJ, (size_t)A.pj_entries * sizeof(float4));
    if (k.hl) need(SLOT_BATCH_FRAME, (size_t)k.C * sizeof(double4));
    if (e != cudaSuccess) return cuda_fail(ctx, e, "scratch allocation (batched)");
    unsigned char *plan = static_cast<unsigned char *>(es.buf[SLOT_BATCH_PLAN]);
    A.planned = reinterpret_cast<BatchKey *>(plan);
    A.nitems = reinterpret_cast<int *>(plan + 64);
    A.head = A.nitems + 1;
    A.split = reinterpret_cast<BatchSplit *>(A.nitems + 2);
    plan += 256;
    A.poff = reinterpret_cast<int64_t *>(plan);
    A.ibase = reinterpret_cast<int64_t *>(plan + b_off);
    A.pjbase = reinterpret_cast<int64_t *>(plan + 2 * b_off);
    A.planned_off = reinterpret_cast<int64_t *>(plan + 3 * b_off);
    A.notes = reinterpret_cast<int *>(plan + 4 * b_off);
    A.weights = reinterpret_cast<int *>(plan + 4 * b_off + b_c);
    A.block = reinterpret_cast<BmBlock *>(plan + 4 * b_off + 2 * b_c);
    A.items = static_cast<int4 *>(es.buf[SLOT_BATCH_ITEMS]);
    A.cp = static_cast<MPart *>(es.buf[SLOT_BATCH_CP]);
    A.pi = static_cast<float4 *>(es.buf[SLOT_BATCH_PI]);
    A.pj = static_cast<float4 *>(es.buf[SLOT_BATCH_PJ]);
    A.err = ctx_err_word(ctx);
    A.wait_ns = ctx_wait_ns(ctx);
    A.pi_len = (int64_t)(es.cap[SLOT_BATCH_PI] / sizeof(float4));
    A.pj_len = (int64_t)(es.cap[SLOT_BATCH_PJ] / sizeof(float4));
    *out = A;
    return NB_OK;
}

// Arguments of a call's kernels; allocates the scratch: per padded block 2 KiB of
// records (4 on two-word positions), 2 of i-side sums and 32 bytes; kItemsPerSm items'
// i-side sums (57 MiB); the j-side sums (batch_pj_entries: 512 MiB, or 265 B for every
// particle beyond the 256th of a cluster). Where that cannot be had, the first alone,
// every pair then being evaluated twice. (10^6 clusters of 32: 5.7 GB.)
nb_status bm_prepare(nb_ctx *ctx, const BatchCall &k, BmArgs *out) {
    ExtState &es = ctx_ext(ctx);
    const int64_t size = k.n_total + k.C * (int64_t)kBlock;
    if (size <= es.batch_max_n) {
        const nb_status st = bm_args(ctx, k, false, out);
        if (st != NB_ERR_OOM) return st;
        es.batch_max_n = size - 1;
    }
    return bm_args(ctx, k, true, out);
}

// One evaluation. `planned`: this call has made one before, so its plan stands and the
// combine has cleared what a plan clears (300 clusters up to 2048, us a step: plain 91.6 ->
// 88, compensated 127 -> 125).
nb_status bm_force(nb_ctx *ctx, const BatchCall &k, BmArgs A, const BatchSource &src, bool planned, float *a, float *p,
                   cudaStream_t st) {
    ExtState &es = ctx_ext(ctx);
    cudaError_t e = cudaSuccess;
    if (!planned) {
        A.fresh = !es.batch_plan;
        e = launch_with_pdl(bm_plan_kernel, dim3(1), dim3(kBmPlanThreads), 0, st, A);
        es.batch_plan = e == cudaSuccess;
    }
    if (e != cudaSuccess) return cuda_fail(ctx, e, "batch plan launch");
    const dim3 blocks((unsigned)(A.cap_padded / kBlock)), threads(kBlock);
    double *const no_v = nullptr;
    const float *const no_a = nullptr;
    if (k.hl) {
        double4 *frame = static_cast<double4 *>(es.buf[SLOT_BATCH_FRAME]);
        if (src.kick) {
            e = launch_with_pdl(batch_kick_drift_kernel, dim3((unsigned)((3 * k.n_total + 255) / 256)), dim3(256), 0, st,
                                src.x64, src.v, src.a, k.n_total, src.dt, src.kick_back);
            if (e != cudaSuccess) return cuda_fail(ctx, e, "leap-frog update launch");
        }
        e = launch_with_pdl(batch_frame_kernel, dim3((unsigned)k.C), dim3(kFrameThreads), 0, st,
                            (const double *)src.x64, k.offsets, (const int64_t *)A.poff, frame);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "batched frame launch");
        e = launch_with_pdl(bm_pack_hl_kernel, blocks, threads, 0, st, A, (const double *)src.x64, src.m,
                            (const double4 *)frame);
    } else if (src.x32) {
        e = launch_with_pdl(bm_pack_kernel<const float, false>, blocks, threads, 0, st, A, src.x32, no_v, no_a, src.m,
                            0.0, 0);
    } else if (src.kick) {
        e = launch_with_pdl(bm_pack_kernel<double, true>, blocks, threads, 0, st, A, src.x64, src.v, src.a, src.m,
                            src.dt, src.kick_back);
    } else {
        e = launch_with_pdl(bm_pack_kernel<double, false>, blocks, threads, 0, st, A, src.x64, no_v, no_a, src.m, 0.0,
                            0);
    }
    if (e != cudaSuccess) return cuda_fail(ctx, e, "batched pack launch");
    const PairVariant v = bm_variant(k);
    {
        TimedLaunch t(ctx, 4, st);
        e = launch_with_pdl(bm_kernel(k), dim3((unsigned)resident_ctas(ctx, v)), dim3(32), v.smem, st, A);
    }
    if (e != cudaSuccess) return cuda_fail(ctx, e, "batched pair kernel launch");
    e = launch_with_pdl(k.hl ? bm_combine_kernel<true> : bm_combine_kernel<false>, blocks, threads, 0, st, A, a, p);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "batched combine launch");
    return NB_OK;
}

nb_status check_batch_args(nb_ctx *ctx, int64_t C, int64_t n_total, int mode) {
    if (C < 0 || n_total < 0) return fail(ctx, NB_ERR_ARG, "n_clusters and n_total must be >= 0");
    if (mode != NB_PLAIN && mode != NB_COMPENSATED) return fail(ctx, NB_ERR_ARG, "unknown mode");
    return NB_OK;
}

}  // namespace

extern "C" {

nb_status nb_force_batched(nb_ctx *ctx, const float *x, const float *m, const int64_t *offsets,
                           int64_t n_clusters, int64_t n_total, const float *eps, float *a, float *p,
                           nb_mode mode, void *stream) {
    if (!ctx) return NB_ERR_ARG;
    nb_status st = check_batch_args(ctx, n_clusters, n_total, mode);
    if (st != NB_OK) return st;
    if (n_clusters == 0 || n_total == 0) return NB_OK;
    if (!x || !m || !offsets || !eps || !a || !p) return fail(ctx, NB_ERR_ARG, "NULL array pointer");
    DeviceGuard g(ctx_device(ctx));
    // One kernel for both modes: its sums are compensated.
    const BatchCall call{offsets, n_clusters, n_total, eps, false};
    BmArgs A;
    if ((st = bm_prepare(ctx, call, &A)) != NB_OK) return st;
    BatchSource src{};
    src.x32 = x;
    src.m = m;
    return bm_force(ctx, call, A, src, false, a, p, static_cast<cudaStream_t>(stream));
}

nb_status nb_leapfrog_batched_step(nb_ctx *ctx, double *x, double *v, const float *m,
                                   const int64_t *offsets, int64_t n_clusters, int64_t n_total,
                                   const float *eps, float *a, float *p, double dt, int nsteps,
                                   int a_valid, nb_mode mode, void *stream) {
    if (!ctx) return NB_ERR_ARG;
    nb_status st = check_batch_args(ctx, n_clusters, n_total, mode);
    if (st != NB_OK) return st;
    if (nsteps < 0) return fail(ctx, NB_ERR_ARG, "nsteps must be >= 0");
    if (!std::isfinite(dt)) return fail(ctx, NB_ERR_ARG, "dt must be finite");
    if (n_clusters == 0 || n_total == 0) return NB_OK;
    if (!x || !v || !m || !offsets || !eps || !a || !p)
        return fail(ctx, NB_ERR_ARG, "NULL array pointer");
    DeviceGuard g(ctx_device(ctx));
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const BatchCall call{offsets, n_clusters, n_total, eps, mode == NB_COMPENSATED};
    BmArgs A;
    if ((st = bm_prepare(ctx, call, &A)) != NB_OK) return st;
    cudaError_t e;
    bool planned = false;
    auto evaluate = [&](int kick, int kick_back) {
        const nb_status rs = bm_force(ctx, call, A, BatchSource{nullptr, x, v, a, m, dt, kick, kick_back}, planned, a,
                                      p, s);
        planned = true;
        return rs;
    };
    auto force = [&]() { return evaluate(0, 0); };
    auto step = [&](int kick_back) { return evaluate(1, kick_back); };

    if (!a_valid && (st = force()) != NB_OK) return st;
    if (nsteps == 0) return NB_OK;
    if ((st = step(0)) != NB_OK) return st;
    const int rest = nsteps - 1;
    if (rest >= 2 && s != nullptr) {
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
        e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "graph capture begin");
        const bool timing = ctx_set_timing(ctx, false);
        nb_status cst = step(1);
        ctx_set_timing(ctx, timing);
        e = cudaStreamEndCapture(s, &graph);
        if (cst != NB_OK) {
            if (graph) cudaGraphDestroy(graph);
            return cst;
        }
        if (e != cudaSuccess) return cuda_fail(ctx, e, "graph capture end");
        e = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "graph instantiate");
        for (int k = 0; k < rest && e == cudaSuccess; ++k) e = cudaGraphLaunch(exec, s);
        cudaGraphExecDestroy(exec);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "graph launch");
    } else {
        for (int k = 0; k < rest; ++k)
            if ((st = step(1)) != NB_OK) return st;
    }
    e = launch_with_pdl(batch_kick_kernel, dim3((unsigned)((3 * n_total + 255) / 256)), dim3(256), 0, s, v,
                        (const float *)a, n_total, dt);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "kick launch");
    return NB_OK;
}

}  // extern "C"
