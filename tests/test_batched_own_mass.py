"""GPU: a particle of infinite or NaN mass does not act on itself in a batch either: its
own results are finite, as nb_force's direct kernels give them, in clusters that are
summed per (i, j) and in clusters whose own blocks are. (What it does to the others is
not finite; where the plain direct kernel gives infinity, compensated sums give NaN.)"""
import numpy as np
import pytest

from test_mutual_parity import batch, ctx, nb, run, run_batch  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mass", [np.inf, np.nan])
@pytest.mark.parametrize("entry", [0, 2])
def test_own_mass_left_out(nb, ctx, entry, mass):
    sizes = [90, 200, 700, 1500]
    x, m, off, eps = batch(sizes)
    m[off[:-1] + 7] = mass
    a, p = run_batch(nb, ctx, (x, m, off, eps), entry)
    try:
        nb.nb_set_tile(ctx, 0, [t for t in nb.nb_list_tiles(0) if not t.fused and not t.packed & 64][0])
        for c in range(len(sizes)):
            s = slice(off[c], off[c + 1])
            a0, p0 = run(nb, ctx, x[s], m[s], eps[c], 0)
            assert np.isfinite(a0[7]).all() and np.isfinite(p0[7]) and np.isfinite(a0).all(1).sum() == 1
            assert np.array_equal(np.isfinite(a0), np.isfinite(a[s])) and np.array_equal(np.isfinite(p0), np.isfinite(p[s])), c
    finally:
        nb.nb_set_tile(ctx, 0, None)
