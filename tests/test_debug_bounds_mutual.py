"""GPU: the kernels that evaluate every pair once under the bounds-checked build
(libnbody_debug.so; test_debug_bounds.py has the idea and the direct kernels): every
mutual shape at the edges of its tiles, panels of rows, batches with several bands and
every kind of weights, the VJP from arrays and from the adjoint's state, and the
potential-only kernels."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_mutual_kernels_under_bounds_checks():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_3659_gb300 import build
    env = dict(os.environ, NB_LIBRARY=build.build(debug=True))
    sel = ("edges or panels or bands or steps or far_and_nonfinite or smaller_calls or larger_scratch or "
           "every_tile or energy or potential or ((trajectory or adjoint) and not plummer16384)")
    files = ["tests/test_mutual_parity.py", "tests/test_panels.py", "tests/test_batched_steps.py",
             "tests/test_captured_force.py", "tests/test_energy_potential.py", "tests/test_vjp_parity.py"]
    r = subprocess.run([sys.executable, "-m", "pytest", *files, "-q", "-m", "gpu", "-k", sel, "-p", "no:cacheprovider"],
                       cwd=ROOT, env=env, capture_output=True, text=True, timeout=1800)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-2000:]
    assert "passed" in r.stdout
