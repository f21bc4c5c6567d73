// nb_batched.cuh -- the work split of the batched kernels that evaluate
// every unordered pair of a cluster once (nb_batched.cu).
//
// Clusters are padded to blocks of kBlock particles. Row b of a cluster is block b
// on the i-side, held by one warp. In a band of consecutive blocks it meets its own
// block and those of other bands for its own side, the later blocks of its band for
// both sides. A band is as long as the batch's longest cluster (nothing is then met
// twice but the own blocks), unless the j-side sums, one float4 per (row, particle of a
// later block of its band), would take more than the scratch set aside: then as long as
// they may be, which the plan finds out, the sizes being on the device.
//
// A row has nt - r blocks to meet (nt blocks in the cluster, r its place in the
// band): its own, the later ones of the band, then the others. It is cut into items
// of `chunk` consecutive blocks, or every block into `parts` items, whichever gives
// the resident warps several items each.
#pragma once

#include <cstdint>

namespace nbk {

constexpr int kBlock = 128;  // particles per block: 4 per lane
constexpr int kTile = 64;    // particles per copy
constexpr int kBlockTiles = kBlock / kTile;
// j-side entries set aside: 512 MiB, or what bands of kMinBand blocks need of clusters of
// that many blocks or more, by the particles beyond the 256th of a cluster (on average:
// the sizes are not known), but no more than the need of a single cluster.
constexpr int64_t kPjEntries = (int64_t)32 << 20;
constexpr int kMinBand = 32;
// Clusters of up to so many blocks are evaluated per (i, j), every block by every row
// (a band of one block): they have few pairs to save (cluster_weights, nb_batched.cu).
constexpr int kDirectBlocks = 2;

__host__ __device__ inline int cluster_band(int band, int64_t nt) { return nt <= kDirectBlocks ? 1 : band; }

// What a plan depends on besides the offsets. A plan made for more j-side entries than
// a call has scratch for must not stand: its sums would go past their buffer.
struct BatchKey {
    int64_t clusters, n_total, want_items, pj_entries;  // clusters -1: no plan
};
__host__ __device__ inline bool same_plan(const BatchKey &a, const BatchKey &b) {
    return a.clusters == b.clusters && a.n_total == b.n_total && a.want_items == b.want_items &&
           a.pj_entries == b.pj_entries;
}

struct BatchSplit {
    int band;          // blocks per band
    int chunk, parts;  // one of them is 1
    // Items of a row with t blocks to meet.
    __host__ __device__ int items(int t) const { return (t + chunk - 1) / chunk * parts; }
    // Items of rows with 1, 2 .. k blocks to meet together.
    __host__ __device__ int64_t below(int64_t k) const {
        const int64_t a = k / chunk;
        return (chunk * (a * (a + 1) / 2) + (k - a * chunk) * (a + 1)) * parts;
    }
    // The first item of row b of a cluster of nt blocks, counted from the
    // cluster's first (b = nt: their number).
    __host__ __device__ int64_t first(int64_t nt, int64_t b) const {
        const int cb = cluster_band(band, nt);
        const int64_t k = b / cb, r = b - k * cb, f = below(nt);
        return (k ? k * (f - below(nt - cb)) : 0) + (r ? f - below(nt - r) : 0);
    }
    // Item k of a row of a cluster of nt blocks, t of them to meet: the met tiles
    // [*v0, *v1). Blocks of the smallest clusters are not parted.
    __host__ __device__ void range(int nt, int t, int k, int *v0, int *v1) const {
        if (parts > 1) {
            constexpr int n = kBlockTiles;
            *v0 = k * (n / parts);
            *v1 = *v0 + n / parts;
            if (nt <= kDirectBlocks) *v1 = k % parts ? *v0 : *v0 + n;
            return;
        }
        const int q = items(t), each = t / q, more = t - each * q;  // the first `more` have one block more
        *v0 = (k * each + (k < more ? k : more)) * kBlockTiles;
        *v1 = *v0 + (each + (k < more)) * kBlockTiles;
    }
};

// The split of a batch whose rows meet `met` blocks in all, `longest` at most, for
// `want` items: at most one item per row more.
__host__ __device__ inline BatchSplit batch_split(int band, int longest, int64_t met, int64_t want) {
    BatchSplit s{band, 1, 1};
    const int64_t chunk = (met + want - 1) / want;
    if (met > want) s.chunk = chunk < longest ? (int)chunk : longest;
    else while (2 * s.parts <= kBlockTiles && 2 * s.parts * met <= want) s.parts *= 2;
    return s;
}
static_assert((kBlockTiles & (kBlockTiles - 1)) == 0, "parts hold equal numbers of tiles");

// Blocks met by all rows of a cluster of nt blocks.
__host__ __device__ inline int64_t batch_met(int band, int64_t nt) { return BatchSplit{band, 1, 1}.first(nt, nt); }

// The v-th block that row b meets.
__host__ __device__ inline int batch_met_block(int band, int nt, int b, int v) {
    band = cluster_band(band, nt);
    const int s0 = b / band * band, s1 = s0 + band < nt ? s0 + band : nt;
    if (v < s1 - b) return b + v;
    const int w = v - (s1 - b);
    return w < s0 ? w : w - s0 + s1;
}

// The v-th tile that row b meets.
__host__ __device__ inline int batch_met_tile(int band, int nt, int b, int v) {
    return batch_met_block(band, nt, b, v / kBlockTiles) * kBlockTiles + v % kBlockTiles;
}

// j-side entries of a cluster of nt blocks.
__host__ __device__ inline int64_t batch_pj_need(int band, int64_t nt) {
    const int64_t cb = cluster_band(band, nt), k = nt / cb, rest = nt - k * cb;
    return (k * (cb * (cb - 1) / 2) + rest * (rest - 1) / 2) * kBlock;
}

// The first j-side entry of row b, counted from the cluster's first (those of the
// particles of its band's later blocks follow).
__host__ __device__ inline int64_t batch_pj_row(int band, int nt, int b) {
    const int cb = cluster_band(band, nt), k = b / cb, s0 = k * cb;  // (32-bit divisions: once per item)
    const int64_t r = b - s0, len = cb < nt - s0 ? cb : nt - s0;
    return (k * ((int64_t)cb * (cb - 1) / 2) + r * len - r * (r + 1) / 2) * kBlock;
}

// Entries set aside for a batch.
inline int64_t batch_pj_entries(int64_t clusters, int64_t n_total) {
    const int64_t most = (n_total + kBlock - 1) / kBlock, one = most * (most - 1) / 2 * kBlock;
    const int64_t beyond = n_total - clusters * (kDirectBlocks * kBlock);
    // (kMinBand - 1) / 2 entries for every one of their particles
    const int64_t bands = beyond * (kMinBand - 1) * kMinBand / (2 * (kMinBand - kDirectBlocks));
    const int64_t want = bands > kPjEntries ? bands : kPjEntries;
    return want < one ? want : one;
}

}  // namespace nbk
