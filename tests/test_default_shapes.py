"""GPU: which kind of shape nb_force takes by size, and that the compensated mode is no
less exact than the direct shapes where both could serve."""
import numpy as np
import pytest

import workloads
from test_mutual_parity import ctx, nb  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


def test_mutual_shapes_by_size(nb):
    with nb.Context(0) as fresh:
        for mode, n, mutual in ((0, 13311, False), (0, 13312, True), (0, 24576, True), (0, 1 << 20, True),
                                (1, 13312, False), (1, 24575, False), (1, 24576, True), (1, 1 << 20, True)):
            assert bool(nb.nb_get_tile(fresh, n, mode).packed & 64) == mutual, (mode, n)


@pytest.mark.parametrize("n", [13312, 20000, 30000])
def test_compensated_force_as_exact_as_the_direct_shapes(nb, ctx, n):
    # 2-norm over 2048 particles, root mean square over four systems; 3% for chance.
    import torch
    eps, rows = 1.0 / 64, np.sort(np.random.default_rng(1).choice(n, 2048, replace=False))
    direct = [t for t in nb.nb_list_tiles(1) if not t.packed & 64 and t.refine == 0 and
              (t.fused == 2 if n < 24576 else (t.threads, t.ipt, t.jtile, t.fused) == (256, 4, 256, 0))]
    error = [0.0, 0.0]
    for seed in range(4):
        x, _, m = workloads.plummer(n, seed=n + 1000 * seed)
        x, m = torch.from_numpy(x.astype(np.float32)).cuda(), torch.from_numpy(m.astype(np.float32)).cuda()
        want, X = [], x.double()
        for k in range(0, len(rows), 64):
            r = torch.from_numpy(rows[k:k + 64]).cuda()
            d = X[r][:, None] - X[None]
            y = (d.square().sum(-1) + eps ** 2).rsqrt()
            y[torch.arange(len(r)), r] = 0
            want.append(((m.double() * y ** 3)[..., None] * d).sum(1))
        want, r = torch.cat(want), torch.from_numpy(rows).cuda()
        for k, tile in enumerate((None, direct[0])):
            a, p = torch.empty_like(x), torch.empty_like(m)
            nb.nb_set_tile(ctx, 1, tile)
            try:
                nb.nb_force(ctx, x, m, n, eps, a, p, 1)
                nb.nb_synchronize(ctx)
            finally:
                nb.nb_set_tile(ctx, 1, None)
            error[k] += float((a[r].double() - want).norm() / want.norm()) ** 2
    assert error[0] <= 1.03 ** 2 * error[1]
