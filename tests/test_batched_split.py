"""CPU: the work split of the batched kernels (csrc/nb_batched.cuh), compiled for the
host: when a kept plan stands for a call."""
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
    # be allocated: the same clusters, particles and items, shorter bands.
    run_host(tmp_path, """
int main() {
    const BatchKey a{100, 29184 * 128, 29184, 32};
    CHECK(same_plan(a, a));
    for (int k = 0; k < 4; ++k) {
        BatchKey b = a;
        (k == 0 ? b.clusters : k == 1 ? b.n_total : k == 2 ? b.want_items : b.max_band) = 1;
        CHECK(!same_plan(a, b) && !same_plan(b, a));
    }
}
""")
