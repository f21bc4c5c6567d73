"""GPU: the register-read rates that bound the kernels which evaluate every pair once
(tests/gpu_probes/fp32_operand_rate.cu): a multiply-add of two distinct registers issues
about every cycle (packed: every two), one of three distinct ones clearly less often."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

PROBE = os.path.join(os.path.dirname(__file__), "gpu_probes", "fp32_operand_rate.cu")


def test_three_distinct_registers_take_longer(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "fp32_operand_rate")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-o", exe, PROBE], check=True,
                   capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    cycles = {name: float(v) for name, v in (line.split() for line in out.splitlines())}
    print(cycles)
    assert 0.95 <= cycles["ffma_two"] <= 1.2 and 1.9 <= cycles["ffma2_two"] <= 2.5, cycles
    assert cycles["ffma_three"] >= 1.3 and cycles["ffma2_three"] >= 3.0, cycles
