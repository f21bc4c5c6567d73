"""CPU: the scratch of the kernels that evaluate every unordered pair once
(csrc/nb_triangle.cuh): what is reserved for n is enough for n
and for every smaller n, in one panel of rows or in several."""
import os
import subprocess

from paper_0904_3659_gb300 import build

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0904_3659_gb300", "csrc")

SOURCE = """
#include <algorithm>
#include <cstdio>
#include "nb_triangle.cuh"
using namespace nbk;
int main() {
    for (int ib : {512, 768, 1024})
        for (int jt : {32, 128})
            for (int64_t most : {1, 100, 5000, 70000}) {
                TriangleScratch before{0, 0, false};
                for (int64_t n = 1; n <= 700 * ib; n += 1 + n / 97) {
                    const Triangle T{(n + jt - 1) / jt, (n + ib - 1) / ib, ib / jt};
                    const TriangleScratch s = triangle_scratch(T, most);
                    int64_t tiles = 1, rows = 1, panels = 0;
                    for (int64_t r0 = 0; r0 < T.nib; ++panels) {
                        const int64_t r1 = T.panel_end(r0, most);
                        tiles = std::max(tiles, T.tiles(r0, r1));
                        rows = std::max(rows, r1 - r0);
                        r0 = r1;
                    }
                    if (tiles > s.tiles || rows > s.rows || (panels > 1) != s.panels || s.tiles < before.tiles ||
                        s.rows < before.rows || s.tiles > std::max(tiles, std::max(most, T.njt))) {
                        std::printf("ib %d jt %d most %ld n %ld\\n", ib, jt, (long)most, (long)n);
                        return 1;
                    }
                    before = s;
                }
            }
}
"""


def test_scratch_covers_every_panel_of_every_smaller_n(tmp_path):
    src = tmp_path / "scratch.cu"
    src.write_text(SOURCE)
    exe = str(tmp_path / "scratch")
    subprocess.run([build.NVCC, *build.ARCH, "-x", "cu", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
