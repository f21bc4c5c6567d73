"""CPU: the work split of the batched kernels (csrc/nb_batched.cuh), compiled for the
host: when a kept plan stands for a call, where the j-side sums go,
and that the items meet everything once."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0904_3659_gb300", "csrc")

HEAD = """
#include <cstdio>
#include <cstdlib>
#include <vector>
#define __host__
#define __device__
#include "nb_batched.cuh"
using namespace nbk;
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\\n", __LINE__, #c); return 1; } } while (0)
"""


def run_host(tmp_path, body):
    src = tmp_path / "split.cpp"
    src.write_text(HEAD + body)
    exe = str(tmp_path / "split")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout


def test_a_plan_stands_for_the_same_key_only(tmp_path):
    # The same batch again, but with the scratch of a call whose j-side sums could not
    # be allocated: the same clusters, particles and items, no j-side sums.
    run_host(tmp_path, """
int main() {
    const BatchKey a{100, 29184 * 128, 29184, 32};
    CHECK(same_plan(a, a));
    for (int k = 0; k < 4; ++k) {
        BatchKey b = a;
        (k == 0 ? b.clusters : k == 1 ? b.n_total : k == 2 ? b.want_items : b.pj_entries) = 1;
        CHECK(!same_plan(a, b) && !same_plan(b, a));
    }
}
""")


def test_j_side_entries_are_apart_and_fit(tmp_path):
    # Every (row, particle of a later block of its band) has an entry of its own inside
    # its cluster's share, for every band length; what is set aside for a batch is
    # bounded by its particles, and by 512 MiB for clusters that need none.
    run_host(tmp_path, """
int main() {
    for (int nt = 1; nt <= 40; ++nt)
        for (int band = 1; band <= 45; ++band) {
            const int64_t need = batch_pj_need(band, nt);
            const int cb = cluster_band(band, nt);
            std::vector<int> used(need, 0);
            int64_t count = 0;
            for (int b = 0; b < nt; ++b) {
                const int end = (b / cb + 1) * cb < nt ? (b / cb + 1) * cb : nt;
                for (int j = b + 1; j < end; ++j)
                    for (int l = 0; l < kBlock; ++l, ++count) {
                        const int64_t at = batch_pj_row(band, nt, b) + (int64_t)(j - b - 1) * kBlock + l;
                        CHECK(at >= 0 && at < need && !used[at]++);
                    }
            }
            CHECK(count == need);
            if (band > 1) CHECK(need >= batch_pj_need(band - 1, nt) || band > nt);
            CHECK(nt > kDirectBlocks || need == 0);
            CHECK(batch_pj_need(1, nt) == 0);
        }
    CHECK(batch_pj_entries(1000000, 32000000) == kPjEntries);
    CHECK(batch_pj_entries(1, 1000) == 8 * 7 / 2 * kBlock);
    CHECK(batch_pj_entries(100, 100) == 0);
    for (int64_t nt : {3, 10, 31, 32, 33, 64, 500})  // bands of 32 blocks in many large clusters
        CHECK(batch_pj_entries(100000, 100000 * nt * kBlock) >= 100000 * batch_pj_need(32, nt));
    for (int64_t n : {1000, 100000, 10000000})
        for (int64_t c : {1, 30, 100000}) CHECK(batch_pj_entries(c, n) <= (n * 17 > kPjEntries ? n * 17 : kPjEntries));
}
""")


def test_items_meet_every_tile_once(tmp_path):
    # Batches of clusters of 0 to 40 blocks in bands of 1 to 45 for few to many wanted
    # items: a row's items meet its own block and the later blocks of its band once
    # (and nothing else of the band), every block of other bands once, and no more items
    # are made than one per row beyond the number wanted.
    run_host(tmp_path, """
int main() {
    unsigned seed = 1;
    auto draw = [&](unsigned n) { seed = seed * 1664525u + 1013904223u; return (int)((seed >> 8) % n); };
    for (int round = 0; round < 600; ++round) {
        const int clusters = 1 + draw(12), band = 1 + draw(45);
        std::vector<int> nt(clusters);
        int64_t met = 0, blocks = 0;
        int longest = 1;
        for (int &n : nt) {
            n = draw(3) ? draw(41) : draw(4);
            met += batch_met(band, n);
            blocks += n;
            longest = n > longest ? n : longest;
        }
        const int64_t want = round % 7 == 0 ? 1 : 1 + draw(4000);
        const BatchSplit split = batch_split(band, longest, met, want);
        int64_t items = 0;
        for (int n : nt) {
            if (n == 0) continue;
            const int cb = cluster_band(band, n);
            int64_t first = 0;
            for (int b = 0; b < n; ++b) {
                CHECK(split.first(n, b) == first);
                const int t = n - b % cb, q = split.items(t), end = (b / cb + 1) * cb;
                first += q;
                std::vector<int> seen(n * kBlockTiles, 0);
                for (int k = 0; k < q; ++k) {
                    int v0, v1;
                    split.range(n, t, k, &v0, &v1);
                    for (int v = v0; v < v1; ++v) {
                        const int tile = batch_met_tile(band, n, b, v);
                        CHECK(tile >= 0 && tile < n * kBlockTiles);
                        ++seen[tile];
                    }
                }
                for (int j = 0; j < n * kBlockTiles; ++j) {
                    const int block = j / kBlockTiles, in_band = block >= b / cb * cb && block < end;
                    CHECK(seen[j] == (in_band && block < b ? 0 : 1));
                }
            }
            CHECK(split.first(n, n) == first);
            items += first;
        }
        CHECK(items <= blocks + want + 1);
    }
}
""")
