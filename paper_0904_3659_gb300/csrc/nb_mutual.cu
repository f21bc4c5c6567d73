// nb_mutual.cu -- Eq. (gravity) (Fujiwara & Nakasato, arXiv:0904.3659, Section
// "Introduction") with every unordered pair evaluated once (nb_mutual.cuh):
// pack -> mutual pair kernel -> combine.
//
// Work. The particles are cut into i-blocks of IB and j-tiles of JT. Row b of
// the triangle is i-block b against the tiles of its own block and of every
// later block. In a tile of its own block a warp meets the groups of the warps
// after it, and its own particles one-sided; the warps before have met theirs.
// The resident CTAs take equal contiguous ranges of the tiles listed row by row
// (nb_triangle.cuh).
//
// Sums. A thread keeps its i-particles' sums for a whole row segment, with
// Kahan compensation across groups of tiles; a segment's sums go to the slot
// c + (b - first row) of `pi`, which no other (CTA c, row b) shares, because c
// or b grows from one segment to the next. The j-side sums of a tile, added
// over the CTA's warps in warp order, go to pj, which holds one float4 per (row,
// particle of the row's tiles). The combine adds, for each particle, its segments in CTA
// order and then its pj entries in row order with compensation. No atomics on
// floats: the result is bit-reproducible for a fixed launch.
//
// pj takes n^2 / (2 IB) float4; above kMutualPartialBytes the rows are done in
// panels of consecutive rows, the combine carrying (sum, carry) per particle
// from panel to panel in the same order of additions.
#include <algorithm>

#include "nb_device.cuh"
#include "nb_ext.h"
#include "nb_internal.h"
#include "nb_mutual.cuh"
#include "nb_triangle.cuh"

namespace nbk {
using namespace nbdev;

// ---------------------------------------------------------------------------
// Pack.
__global__ void mutual_pack_f32_kernel(const float *__restrict__ x, const float *__restrict__ m,
                                       int64_t n, int64_t npad, MPart *__restrict__ cp,
                                       float eps, int *__restrict__ notes) {
    pdl_wait_then_release();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    MPart v = mutual_padding();
    if (i < n) v = make_float4(-x[3 * i], -x[3 * i + 1], -x[3 * i + 2], -0.5f * m[i]);
    mutual_note(i < n, v, -0.5f * m[0], eps, notes);
    if (i < npad) cp[i] = v;
}

// ---------------------------------------------------------------------------
// WARPS x 32 threads, P packed i-pairs per thread, JT-particle j-tiles in
// STAGES buffers, UNR the unroll of the j loop (16 no longer fits the instruction
// cache: 25% slower), MINB the CTAs per SM that the registers are held to, POT
// with the potential, HL on two-word positions.
// W: the form of the weights. From n = 24576 (18432 on two-word positions) the three
// forms are three kernels;
// all are launched and those not meant return at once (the choice is the pack's,
// on the device): with the loops in one kernel (kAny) each of them runs 5-8%
// slower, the registers being allocated for the worst. Below, the two launches
// saved are worth more.
template <int WARPS, int P, int JT, int STAGES, int UNR, int MINB, bool POT, bool HL, int W>
__global__ void __launch_bounds__(WARPS * 32, MINB) mutual_kernel(const MutualArgs A) {
    constexpr int THREADS = WARPS * 32;
    constexpr int IB = 64 * P * WARPS;
    constexpr int TPB = IB / JT;
    constexpr int RS = HL ? kHLRecords : 1;
    constexpr uint32_t TILE_BYTES = JT * RS * sizeof(MPart);
    constexpr int NC = POT ? 4 : 3;
    // Tiles between two compensated additions to the running sums: 128 j-particles with
    // 32-particle tiles, the direct kernels' tiles on FP64 state at those n (with 256 the
    // error of p against FP64 was 1.06 to 1.12 times theirs from N = 12000 to 30000, as it
    // is 0.94 to 0.99; N = 20000 194.3 -> 194.8 us a step), 256 with larger ones.
    constexpr int FOLD = JT <= 32 ? 128 / JT : JT >= 256 ? 1 : 256 / JT;
    static_assert(IB % JT == 0 && JT % 32 == 0, "whole tiles per block, whole groups per tile");
    static_assert(TILE_BYTES % 16 == 0, "bulk copies move multiples of 16 bytes");

    // Shared memory: [STAGES tiles][2 x WARPS x JT j-side sums][running sums,
    // carries][barriers][issue records]
    extern __shared__ __align__(128) unsigned char smem[];
    MPart *tiles = reinterpret_cast<MPart *>(smem);
    float4 *jsum = reinterpret_cast<float4 *>(smem + (size_t)STAGES * TILE_BYTES);
    float2 *ssum = reinterpret_cast<float2 *>(jsum + 2 * WARPS * JT);
    float2 *scmp = ssum + 4 * P * THREADS;
    uint64_t *full = reinterpret_cast<uint64_t *>(scmp + 4 * P * THREADS);
    int *issued_at = reinterpret_cast<int *>(full + STAGES);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // The packed particles are ready. The combine's blocks, resident early, slow the
    // kernel down at small n (compensated step, N = 4096 32.0 -> 30.1 us, N = 16384
    // 140 -> 139); with a kernel per form the next one is released (N = 65536 1287
    // against 1294 us).
    if (W == kAny) pdl_wait();
    else pdl_wait_then_release();
    const int weights = mutual_weights(__ldcg(A.notes) | (A.wide_eps ? kNoteWide : 0));
    if (W != kAny && W != weights) return;
    const int64_t c = blockIdx.x;
    if (c == 0 && tid == 0) *A.weights = weights;  // for the combine
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

    int64_t pb = b, pt = t;  // thread 0: the next tile to copy
    auto issue = [&](int kk) {
        const int64_t tile = pt;
        if (++pt == A.njt) {
            ++pb;
            pt = pb * TPB;
        }
        if (first + kk == A.fault_unit) return;  // test hook: this copy never happens
        if (!NB_IN(A.err, 40, (tile + 1) * JT <= A.npad)) return;
        const int s = kk % STAGES;
        issued_at[s] = kk;
        mbar_arrive_expect_tx(&full[s], TILE_BYTES);
        bulk_g2s(tiles + (size_t)s * JT * RS, A.cp + tile * JT * RS, TILE_BYTES, &full[s]);
    };
    if (tid == 0)
        for (int kk = 0; kk < count && kk < STAGES - 1; ++kk) issue(kk);

    const float2 eps2 = splat2(A.eps2), zero2 = splat2(0.f);
    MutualI<P, HL> I;
    float2 acc[P][4];
#pragma unroll
    for (int q = 0; q < P; ++q)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[q][r] = zero2;
    int held = 0;  // tiles in acc since the last fold

    // The sums of the tiles in acc enter the running sums (Kahan: the true
    // value is sum - carry).
    auto fold = [&]() {
#pragma unroll
        for (int q = 0; q < P; ++q)
#pragma unroll
            for (int r = 0; r < NC; ++r) {
                const int k = (4 * q + r) * THREADS + tid;
                const float2 s0 = ssum[k];
                const float2 y = add2(acc[q][r], neg2(scmp[k]));
                const float2 v = add2(s0, y);
                scmp[k] = add2(add2(v, neg2(s0)), neg2(y));
                ssum[k] = v;
                acc[q][r] = zero2;
            }
        held = 0;
    };
    auto flush = [&](int64_t row) {
        fold();
        const int64_t off = (c + row - A.r0) * 2 * (int64_t)IB;
        if (!NB_IN(A.err, 41, off >= 0 && off + 2 * IB <= A.pi_len)) return;
        float4 *dst = A.pi + off + warp * 64 * P + lane;
#pragma unroll
        for (int q = 0; q < P; ++q) {
            float2 s[4], k[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                s[r] = r < NC ? ssum[(4 * q + r) * THREADS + tid] : zero2;
                k[r] = r < NC ? scmp[(4 * q + r) * THREADS + tid] : zero2;
            }
            dst[64 * q] = make_float4(s[0].x, s[1].x, s[2].x, s[3].x);
            dst[64 * q + 32] = make_float4(s[0].y, s[1].y, s[2].y, s[3].y);
            dst[IB + 64 * q] = make_float4(k[0].x, k[1].x, k[2].x, k[3].x);
            dst[IB + 64 * q + 32] = make_float4(k[0].y, k[1].y, k[2].y, k[3].y);
        }
    };
    // The j-side sums of the tile before (its warps' in warp order), to pj.
    int64_t put_at = 0;
    auto put = [&](int buf) {
        if (!NB_IN(A.err, 42, put_at + JT <= A.pj_len)) return;
        for (int j = tid; j < JT; j += THREADS) {
            float4 v = jsum[(buf * WARPS) * JT + j];
#pragma unroll
            for (int w = 1; w < WARPS; ++w) {
                const float4 u = jsum[(buf * WARPS + w) * JT + j];
                v = make_float4(__fadd_rn(v.x, u.x), __fadd_rn(v.y, u.y), __fadd_rn(v.z, u.z),
                                __fadd_rn(v.w, u.w));
            }
            A.pj[put_at + j] = v;
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
                if (!NB_IN(A.err, 43, i1 < A.npad)) i0 = i1 = 0;
                const float4 u = A.cp[i0 * RS], w = A.cp[i1 * RS];
                I.x[q] = make_float2(-u.x, -w.x);
                I.y[q] = make_float2(-u.y, -w.y);
                I.z[q] = make_float2(-u.z, -w.z);
                I.hm[q] = make_float2(u.w, w.w);
                if (W == kProduct || (W == kAny && weights == kProduct))
                    I.hm[q] = make_float2(mutual_scale(u.w, A.cp[0].w, A.eps), mutual_scale(w.w, A.cp[0].w, A.eps));
                if constexpr (HL) {
                    const float4 ul = A.cp[i0 * RS + 1], wl = A.cp[i1 * RS + 1];
                    I.lx[q] = make_float2(-ul.x, -wl.x);
                    I.ly[q] = make_float2(-ul.y, -wl.y);
                    I.lz[q] = make_float2(-ul.z, -wl.z);
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    ssum[(4 * q + r) * THREADS + tid] = zero2;
                    scmp[(4 * q + r) * THREADS + tid] = zero2;
                }
            }
        }

        const int s = k % STAGES;
        if (!mbar_wait_bounded(&full[s], (uint32_t)((k / STAGES) & 1), A.wait_ns)) {
            bad = 1;
            continue;
        }
        const MPart *tile = tiles + (size_t)s * JT * RS;
        put_at = (T.lin(b) - pj0 + t - b * TPB) * JT;
        float4 *dst = jsum + ((k & 1) * WARPS + warp) * JT + lane;
        // In the own block: the warp's own groups one-sided, others by met().
        const int64_t own = (t - b * TPB) * (JT / 32) - warp * 2 * P;
#pragma unroll 1
        for (int g = 0; g < JT / 32; ++g) {
            const MPart *G = tile + g * 32 * RS;
            float ja[4] = {0.f, 0.f, 0.f, 0.f};
            const int o = (int)own + g;  // the group, counted from the warp's first
            if (t >= (b + 1) * TPB || met<WARPS, 2 * P>(o, warp, b & 1))
                run_group<P, UNR, POT, HL, W>(weights, G, lane, I, acc, ja, eps2);
            else if (o >= 0 && o < 2 * P)
                run_self<P, POT, HL, W>(weights, G, lane, o, I, acc, eps2);
            dst[32 * g] = make_float4(ja[0], ja[1], ja[2], ja[3]);
        }
        if (++held == FOLD) fold();
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

// ---------------------------------------------------------------------------
// Combine.
// 32 particles per block, one per lane, and their entries (pj of the rows, then
// the segments of their own row in CTA order) in equal contiguous shares for the
// warps, whose sums are then added in warp order: a particle of the first row has
// up to a hundred segments at small n, and reading them one after the other took
// 17 us at N = 3001.
constexpr int kCombineWarps = 8;

__global__ void __launch_bounds__(32 * kCombineWarps) mutual_combine_kernel(const MutualArgs A, const MutualOut O) {
    __shared__ float part[kCombineWarps][8][32];
    pdl_wait_then_release();
    if (O.last && blockIdx.x == 0 && threadIdx.x == 0) *A.notes = 0;  // for the next call's pack
    constexpr int K = 8;  // loads in flight
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = blockIdx.x * (int64_t)32 + lane;  // below the padded count
    const int ib = O.ib;
    const int64_t b = blockIdx.x * (int64_t)32 / ib, w = i - b * ib;
    float S[4] = {0.f, 0.f, 0.f, 0.f}, E[4] = {0.f, 0.f, 0.f, 0.f};
    // j-side sums (of the opposite sign) of rows r0 .. below r1, up to its own.
    const int64_t rend = b + 1 < A.r1 ? b + 1 : A.r1;
    const int rows = rend > A.r0 ? (int)(rend - A.r0) : 0;
    int c0 = 0, segs = 0;
    if (b >= A.r0 && b < A.r1) {  // (clamped: after a timeout the two words may be stale)
        c0 = max(A.row_first[b], 0);
        segs = max(min(A.row_last[b], A.grid - 1) - c0 + 1, 0);
    }
    const int e0 = (int)((int64_t)(rows + segs) * warp / kCombineWarps);
    const int e1 = (int)((int64_t)(rows + segs) * (warp + 1) / kCombineWarps);
    // Row r's entry of i is (lin(r) - lin(r0)) JT + i - r ib; the next row's is
    // (njt - r tpb) JT - ib further.
    const Triangle T{A.njt, A.nib, ib / O.jt};
    int64_t at = (T.lin(A.r0 + e0) - T.lin(A.r0)) * O.jt + i - (A.r0 + e0) * ib;
    int64_t step = (A.njt - (A.r0 + e0) * T.tpb) * O.jt - ib;
    for (int e = e0; e < e1 && e < rows; e += K) {
        float4 v[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (e + k < e1 && e + k < rows && NB_IN(A.err, 44, at >= 0 && at < A.pj_len)) v[k] = __ldcg(A.pj + at);
            at += step;
            step -= ib;
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float h[4] = {-v[k].x, -v[k].y, -v[k].z, v[k].w};
            comp_add(S, E, h);  // (past the end: zeros)
        }
    }
    // Segments: sum - carry.
    for (int e = max(e0, rows); e < e1; e += K / 2) {
        float4 hi[K / 2], lo[K / 2];
#pragma unroll
        for (int k = 0; k < K / 2; ++k) {
            const int64_t o = (c0 + e + k - rows + b - A.r0) * 2 * (int64_t)ib + w;
            hi[k] = lo[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (e + k >= e1 || !NB_IN(A.err, 45, o >= 0 && o + ib < A.pi_len)) continue;
            hi[k] = __ldcg(A.pi + o);
            lo[k] = __ldcg(A.pi + o + ib);
        }
#pragma unroll
        for (int k = 0; k < K / 2; ++k) {
            const float h[4] = {hi[k].x, hi[k].y, hi[k].z, hi[k].w};
            const float l[4] = {lo[k].x, lo[k].y, lo[k].z, lo[k].w};
            comp_add(S, E, h);
#pragma unroll
            for (int r = 0; r < 4; ++r) E[r] = __fsub_rn(E[r], l[r]);
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        part[warp][r][lane] = S[r];
        part[warp][4 + r][lane] = E[r];
    }
    __syncthreads();
    if (warp > 0 || i >= O.n) return;
#pragma unroll
    for (int r = 0; r < 4; ++r) S[r] = E[r] = 0.f;
    if (A.r0 > 0) {
        const float4 s = O.state[2 * i], e = O.state[2 * i + 1];
        S[0] = s.x, S[1] = s.y, S[2] = s.z, S[3] = s.w;
        E[0] = e.x, E[1] = e.y, E[2] = e.z, E[3] = e.w;
    }
    for (int q = 0; q < kCombineWarps; ++q) {
        const float h[4] = {part[q][0][lane], part[q][1][lane], part[q][2][lane], part[q][3][lane]};
        comp_add(S, E, h);
#pragma unroll
        for (int r = 0; r < 4; ++r) E[r] = __fadd_rn(E[r], part[q][4 + r][lane]);
    }
    if (!O.last) {
        O.state[2 * i] = make_float4(S[0], S[1], S[2], S[3]);
        O.state[2 * i + 1] = make_float4(E[0], E[1], E[2], E[3]);
        return;
    }
    // The factors that the weights left out: the mass (kEqual; the first record
    // holds -m/2), 1 / (c m_i) (kProduct), -2 (kWide).
    const int weights = *A.weights;
    const int rs = O.hl ? kHLRecords : 1;
    const float hm0 = A.cp[0].w, f = weights == kProduct ? mutual_scale(A.cp[i * rs].w, hm0, A.eps) : hm0;
    float v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) v[r] = mutual_result(weights, S[r], E[r], f);
    if (O.a) {
        O.a[3 * i + 0] = v[0];
        O.a[3 * i + 1] = v[1];
        O.a[3 * i + 2] = v[2];
    }
    if (O.p) O.p[i] = v[3];
}

// ---------------------------------------------------------------------------
// Compiled shapes.
template <int WARPS, int P, int JT, int STAGES, bool HL>
constexpr size_t mutual_smem() {
    return (size_t)STAGES * JT * (HL ? kHLRecords : 1) * sizeof(MPart) + (size_t)2 * WARPS * JT * sizeof(float4) +
           (size_t)2 * 4 * P * WARPS * 32 * sizeof(float2) + (size_t)STAGES * (sizeof(uint64_t) + sizeof(int));
}

// Unroll of the j loop per form (8 for equal masses). On FP64 state the whole run of 8
// steps, against 4 and 2: leap-frog step with the potential, N = 65536, unequal masses
// 1941 -> 1887 us, with massless tracers 2172 -> 2055; without it 1819 -> 1714, 2023 ->
// 1823.
template <bool HL>
constexpr int kUnrollProduct = HL ? 8 : 4;
template <bool HL>
constexpr int kUnrollWide = HL ? 8 : 2;

template <int W, int P, int J, int S, int M, bool POT, bool HL>
static cudaError_t launch_mutual(MutualArgs a, const int (&grid)[3], size_t smem, cudaStream_t st) {
    a.grid = grid[kWide];
    cudaError_t e = launch_with_pdl(mutual_kernel<W, P, J, S, kUnrollWide<HL>, M, POT, HL, kWide>, dim3((unsigned)a.grid),
                                    dim3(W * 32), smem, st, a);
    a.grid = grid[kProduct];
    if (e == cudaSuccess)
        e = launch_with_pdl(mutual_kernel<W, P, J, S, kUnrollProduct<HL>, M, POT, HL, kProduct>, dim3((unsigned)a.grid),
                            dim3(W * 32), smem, st, a);
    a.grid = grid[kEqual];
    if (e == cudaSuccess)
        e = launch_with_pdl(mutual_kernel<W, P, J, S, 8, M, POT, HL, kEqual>, dim3((unsigned)a.grid),
                            dim3(W * 32), smem, st, a);
    return e;
}

template <int W, int P, int J, int S, int M, bool POT, bool HL>
static cudaError_t launch_mutual_any(MutualArgs a, const int (&grid)[3], size_t smem, cudaStream_t st) {
    a.grid = grid[0];
    return launch_with_pdl(mutual_kernel<W, P, J, S, 4, M, POT, HL, kAny>, dim3((unsigned)a.grid), dim3(W * 32), smem,
                           st, a);
}

// The three forms in one kernel.
#define NB_MUTUAL_ANY(W, P, J, S, M, POT, HL)                                               \
    {W * 32, 64 * P * W, J, HL, POT,                                                        \
     {(const void *)mutual_kernel<W, P, J, S, 4, M, POT, HL, kAny>,                         \
      (const void *)mutual_kernel<W, P, J, S, 4, M, POT, HL, kAny>,                         \
      (const void *)mutual_kernel<W, P, J, S, 4, M, POT, HL, kAny>},                        \
     mutual_smem<W, P, J, S, HL>(), launch_mutual_any<W, P, J, S, M, POT, HL>}
#define NB_MUTUAL(W, P, J, S, M, POT, HL)                                               \
    {W * 32, 64 * P * W, J, HL, POT,                                                        \
     {(const void *)mutual_kernel<W, P, J, S, 8, M, POT, HL, kEqual>,                       \
      (const void *)mutual_kernel<W, P, J, S, kUnrollProduct<HL>, M, POT, HL, kProduct>,                     \
      (const void *)mutual_kernel<W, P, J, S, kUnrollWide<HL>, M, POT, HL, kWide>},                       \
     mutual_smem<W, P, J, S, HL>(), launch_mutual<W, P, J, S, M, POT, HL>}

// [kMutualSmall, Mid, Large][potential or not][HL]
static const MutualShape kMutualShapes[kMutualSizes][2][2] = {
    {{NB_MUTUAL_ANY(4, 4, 32, 3, 3, true, false), NB_MUTUAL_ANY(4, 3, 32, 3, 3, true, true)},
     {NB_MUTUAL_ANY(4, 4, 32, 3, 3, false, false), NB_MUTUAL_ANY(4, 3, 32, 3, 3, false, true)}},
    {{NB_MUTUAL(4, 4, 32, 3, 3, true, false), NB_MUTUAL(4, 3, 32, 3, 3, true, true)},
     {NB_MUTUAL(4, 4, 32, 3, 3, false, false), NB_MUTUAL(4, 3, 32, 3, 3, false, true)}},
    {{NB_MUTUAL(4, 4, 128, 3, 3, true, false), NB_MUTUAL(4, 3, 128, 3, 3, true, true)},
     {NB_MUTUAL(4, 4, 128, 3, 3, false, false), NB_MUTUAL(4, 3, 128, 3, 3, false, true)}},
};
#undef NB_MUTUAL
#undef NB_MUTUAL_ANY

const MutualShape &mutual_shape(int size, bool pot, bool hl) {
    return kMutualShapes[size][pot ? 0 : 1][hl ? 1 : 0];
}

}  // namespace nbk

using namespace nbk;

namespace nbx {

namespace {

// Resident CTAs of the kernel for weights w.
int shape_resident(nb_ctx *ctx, const MutualShape &s, int w) {
    PairVariant v{};
    v.tile.threads = s.threads;
    v.kernel = s.kernel[w];
    v.smem = s.smem;
    return resident_ctas(ctx, v);
}

int most_resident(nb_ctx *ctx, const MutualShape &s) {
    return std::max({shape_resident(ctx, s, 0), shape_resident(ctx, s, 1), shape_resident(ctx, s, 2)});
}

int64_t blocks_of(const MutualShape &s, int64_t n) { return (n + s.ib - 1) / s.ib; }

Triangle triangle(const MutualShape &s, int64_t n) {
    return Triangle{(n + s.jt - 1) / s.jt, blocks_of(s, n), s.ib / s.jt};
}

// Tiles whose j-side sums fit the bound on pj.
int64_t panel_tiles(const MutualShape &s) { return (int64_t)(kMutualPartialBytes / sizeof(float4)) / s.jt; }

}  // namespace

int64_t mutual_npad(const MutualShape &s, int64_t n) { return round_up(std::max<int64_t>(n, 1), s.ib); }

nb_status mutual_reserve(nb_ctx *ctx, const MutualShape &s, int64_t n, MutualUser user) {
    ExtState &es = ctx_ext(ctx);
    auto need = [&](MutualPart part, size_t bytes) {
        const int k = mutual_slot(user, part);
        return ensure_buffer(&es.buf[k], &es.cap[k], bytes);
    };
    const Triangle T = triangle(s, n);
    const TriangleScratch size = triangle_scratch(T, panel_tiles(s));
    const int64_t pi = (most_resident(ctx, s) + size.rows) * 2 * s.ib, pj = size.tiles * s.jt;
    const size_t records = s.hl ? kHLRecords : 1;
    cudaError_t e = need(kPartCp, (size_t)mutual_npad(s, n) * records * sizeof(MPart));
    if (e == cudaSuccess) e = need(kPartPi, (size_t)pi * sizeof(float4));
    if (e == cudaSuccess) e = need(kPartPj, (size_t)pj * sizeof(float4));
    if (e == cudaSuccess) e = need(kPartRows, (size_t)2 * T.nib * sizeof(int));
    if (e == cudaSuccess && size.panels) e = need(kPartState, (size_t)n * 2 * sizeof(float4));
    if (e == cudaSuccess && !es.buf[SLOT_MUTUAL_NOTES]) {
        e = ensure_buffer(&es.buf[SLOT_MUTUAL_NOTES], &es.cap[SLOT_MUTUAL_NOTES], 2 * sizeof(int));
        if (e == cudaSuccess) e = cudaMemset(es.buf[SLOT_MUTUAL_NOTES], 0, 2 * sizeof(int));
        if (e == cudaSuccess) e = cudaDeviceSynchronize();
    }
    if (e == cudaSuccess) return NB_OK;
    if (e == cudaErrorMemoryAllocation) es.mutual_max_n = std::min(es.mutual_max_n, n - 1);
    return cuda_fail(ctx, e, "scratch allocation (mutual pair sums)");
}

MPart *mutual_records(nb_ctx *ctx, MutualUser user) {
    return static_cast<MPart *>(ctx_ext(ctx).buf[mutual_slot(user, kPartCp)]);
}
int *mutual_notes(nb_ctx *ctx) { return static_cast<int *>(ctx_ext(ctx).buf[SLOT_MUTUAL_NOTES]); }

nb_status run_mutual(nb_ctx *ctx, const MutualShape &s, const float *x, const float *m, int64_t n, float eps,
                     float *a, float *p, cudaStream_t st) {
    const MutualUser user = x ? kMutualForce : kMutualFp64;
    cudaError_t e;
    if (x) {
        TimedLaunch t(ctx, 0, st);
        const int64_t npad = mutual_npad(s, n);
        e = launch_with_pdl(mutual_pack_f32_kernel, dim3((unsigned)mutual_pack_blocks(npad)),
                            dim3(kMutualPackThreads), 0, st, x, m, n, npad, mutual_records(ctx, user), eps, mutual_notes(ctx));
        if (e != cudaSuccess) return cuda_fail(ctx, e, "pack kernel launch");
    }
    ExtState &es = ctx_ext(ctx);
    const Triangle T = triangle(s, n);
    MutualArgs A{};
    auto part = [&](MutualPart k) { return es.buf[mutual_slot(user, k)]; };
    A.cp = mutual_records(ctx, user);
    A.pi = static_cast<float4 *>(part(kPartPi));
    A.pj = static_cast<float4 *>(part(kPartPj));
    A.row_first = static_cast<int *>(part(kPartRows));
    A.row_last = A.row_first + T.nib;
    A.notes = mutual_notes(ctx);
    A.weights = mutual_notes(ctx) + 1;
    // eps outside [1 / kMutualRange, kMutualRange]: WIDE whatever the positions.
    A.wide_eps = !(eps >= 1.f / kMutualRange && eps <= kMutualRange);
    A.err = ctx_err_word(ctx);
    A.njt = T.njt;
    A.nib = T.nib;
    A.eps = eps;
    A.eps2 = eps * eps;
    A.fault_unit = ctx_fault_unit(ctx);
    A.wait_ns = ctx_wait_ns(ctx);
    A.npad = mutual_npad(s, n);
    A.pi_len = (int64_t)(es.cap[mutual_slot(user, kPartPi)] / sizeof(float4));
    A.pj_len = (int64_t)(es.cap[mutual_slot(user, kPartPj)] / sizeof(float4));
    MutualOut O{};
    O.state = static_cast<float4 *>(part(kPartState));
    O.n = n;
    O.ib = s.ib;
    O.jt = s.jt;
    O.hl = s.hl;
    for (int64_t r0 = 0; r0 < T.nib;) {
        const int64_t r1 = T.panel_end(r0, panel_tiles(s));
        A.r0 = r0;
        A.r1 = r1;
        A.tiles = T.tiles(r0, r1);
        int grid[3];
        for (int w = 0; w < 3; ++w)
            grid[w] = triangle_grid(A.tiles, shape_resident(ctx, s, w));
        A.grid = most_resident(ctx, s);  // bounds the combine's reads
        {
            TimedLaunch t(ctx, 1, st, s.kernel[0] == s.kernel[1] ? 1 : 3);
            e = s.launch(A, grid, s.smem, st);
        }
        if (e != cudaSuccess) return cuda_fail(ctx, e, "mutual pair kernel launch");
        O.last = r1 == T.nib;
        O.a = O.last ? a : nullptr;
        O.p = O.last ? p : nullptr;
        {
            TimedLaunch t(ctx, 2, st);
            e = launch_with_pdl(mutual_combine_kernel,
                                dim3((unsigned)((n + 31) / 32)), dim3(32 * kCombineWarps), 0, st, A, O);
        }
        if (e != cudaSuccess) return cuda_fail(ctx, e, "combine kernel launch");
        r0 = r1;
    }
    return NB_OK;
}

}  // namespace nbx
