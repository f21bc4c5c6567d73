// nb_triangle.cuh -- the work listing shared by the kernels that evaluate every
// unordered pair once (nb_mutual.cu, nb_vjp_mutual.cu): the triangle of (i-block,
// j-tile) units, and the compensated addition of their combines.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace nbk {

// Row b is i-block b against the tiles of its own block and of every later one.
// lin(b) is the linear index of its first tile, counted row by row from row 0,
// with `tpb` tiles per block and `njt` in all. All tiles count alike: one of the
// own block has half the work of another, but its slowest warp has as much, and a
// CTA meets at a barrier after every tile (force, N = 24576, equal masses: 212 us,
// 255 with own-block tiles at 5/8 of the cost, 220 at 12/8).
struct Triangle {
    int64_t njt, nib;
    int tpb;
    __host__ __device__ int64_t lin(int64_t b) const { return b * njt - tpb * (b * (b - 1) / 2); }
    __host__ __device__ int64_t tiles(int64_t r0, int64_t r1) const { return lin(r1) - lin(r0); }
    // The end of the panel that starts at row r0: as many rows as have at most
    // `most` tiles, at least one.
    int64_t panel_end(int64_t r0, int64_t most) const {
        int64_t lo = r0 + 1, hi = nib;
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) / 2;
            if (tiles(r0, mid) <= most) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    }
    // Row and tile of the u-th tile of rows [r0, r1); (r1, r1 tpb) past the end.
    __device__ void locate(int64_t u, int64_t r0, int64_t r1, int64_t *b, int64_t *t) const {
        u += lin(r0);
        int64_t lo = r0, hi = r1;  // the largest row with lin(row) <= u
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) / 2;
            if (lin(mid) <= u) lo = mid;
            else hi = mid - 1;
        }
        *b = lo;
        *t = lo * tpb + (lo < r1 ? u - lin(lo) : 0);
    }
};

// CTAs for `tiles` tiles on `resident` places: no more than it takes for none to
// have more tiles than ceil(tiles / resident) (VJP, N = 4096, 576 tiles: 29.5 us
// with 288 CTAs of two tiles, 34.6 with 456 of one or two).
inline int triangle_grid(int64_t tiles, int resident) {
    const int64_t each = (tiles + resident - 1) / resident;
    return (int)((tiles + each - 1) / each);
}

// Scratch for the triangle in panels of at most `most` tiles: tiles of a panel, rows of
// one, and whether there are several. It is enough for every smaller triangle of the
// same blocks too: one in a single panel may have more tiles or rows than the panels of
// a larger one have.
struct TriangleScratch {
    int64_t tiles, rows;
    bool panels;
};
inline TriangleScratch triangle_scratch(const Triangle &T, int64_t most) {
    if (T.tiles(0, T.nib) <= most) return {T.tiles(0, T.nib), T.nib, false};
    int64_t rows = 1;  // the most whose tiles, those of the end of a triangle, can be `most`
    while (T.tpb * (rows * (rows + 1) / 2) + rows + 1 <= most) ++rows;
    return {most > T.njt ? most : T.njt, rows, T.nib > 1};
}

// Whether, inside an i-block, warp `w` of WARPS (each with G groups) meets the
// group `o`, counted from its own first group, for both sides: those of the
// next warp, and two of the warps those of the warp after that (the other two
// in odd rows), so that every pair of warps meets once.
template <int WARPS, int G>
__device__ __forceinline__ bool met(int o, int w, bool odd) {
    static_assert(WARPS == 4, "written for four warps");
    if (o < 0) o += WARPS * G;
    return (o >= G && o < 2 * G) || (o >= 2 * G && o < 3 * G && (w == 0 || w == 3) != odd);
}

// (S, E) += h: Knuth's error-free sum, the lost low part kept in E.
template <int N>
__device__ __forceinline__ void comp_add(float (&S)[N], float (&E)[N], const float (&h)[N]) {
#pragma unroll
    for (int r = 0; r < N; ++r) {
        const float v = __fadd_rn(S[r], h[r]);  // TwoSum
        const float bp = __fsub_rn(v, S[r]);
        const float e = __fadd_rn(__fsub_rn(S[r], __fsub_rn(v, bp)), __fsub_rn(h[r], bp));
        S[r] = v;
        E[r] = __fadd_rn(E[r], e);
    }
}

}  // namespace nbk
