"""GPU: the VJP's mutual shapes are no less exact than the direct shapes that they stand
in for (with a gradient on p two packed pairs per thread and 128-particle tiles, without
it one pair and 64-particle tiles). The errors against FP64 are
2-norms over 1024 particles, root mean squares over six systems; 5% is allowed for
what is left to chance (both errors are sums of some 10^7 independent roundings, but the
largest terms, of the closest pairs, count most)."""
import numpy as np
import pytest

import workloads
from test_mutual_parity import ctx, nb  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


def exact_rows(x, m, eps, ga, gp, rows):
    """gx, gm of the rows in FP64 (the formulas of test_vjp_parity.py)."""
    import torch
    X, M, G, P = (t.double() for t in (x, m, ga, gp))
    gx, gm = [], []
    for k in range(0, len(rows), 64):
        r = torch.from_numpy(rows[k:k + 64]).cuda()
        d = X[r][:, None] - X[None]
        y = (d.square().sum(-1) + float(np.float32(eps)) ** 2).rsqrt()
        y[torch.arange(len(r)), r] = 0
        rk, rl, y3 = (d * G[r][:, None]).sum(-1), (d * G[None]).sum(-1), y ** 3
        c = 3 * y ** 5 * (M[r][:, None] * rl - M * rk) - y3 * (P[r][:, None] * M + M[r][:, None] * P)
        gx.append((c[..., None] * d).sum(1) + G[r] * (M * y3).sum(1)[:, None] - M[r][:, None] * (y3 @ G))
        gm.append((P * y).sum(1) - (rl * y3).sum(1))
    return torch.cat(gx), torch.cat(gm)


def compare(nb, ctx, n, with_gp, shape):
    import torch
    eps = 1.0 / 64
    direct = [t for t in nb.nb_list_vjp_tiles() if (t.threads, t.ipt, t.jtile, t.minblocks, t.release) == shape]
    assert len(direct) == 1
    error = [0.0, 0.0]  # of the built-in shape, a mutual one, and of the direct one
    assert nb.nb_get_vjp_tile(ctx, n).packed & 64
    for seed in range(6):
        x, _, m = workloads.plummer(n, seed=1000 * seed + n)
        rng = np.random.default_rng(seed)
        x, m, ga, gp = (torch.from_numpy(v.astype(np.float32)).cuda()
                        for v in (x, m, rng.normal(size=(n, 3)), with_gp * rng.normal(size=n)))
        rows = workloads.sample_rows(n, 1024, seed)
        _, want = exact_rows(x, m, eps, ga, gp, rows)
        for k, tile in enumerate((None, direct[0])):
            gx, gm = torch.empty_like(x), torch.empty_like(m)
            nb.nb_set_vjp_tile(ctx, tile)
            try:
                nb.nb_force_vjp(ctx, x, m, n, eps, ga, gp if with_gp else None, gx, gm)
                nb.nb_synchronize(ctx)
            finally:
                nb.nb_set_vjp_tile(ctx, None)
            e = gm[torch.from_numpy(rows).cuda()].double() - want
            error[k] += float(e.norm() / want.norm()) ** 2
    assert error[0] <= 1.05 ** 2 * error[1]


@pytest.mark.parametrize("n", [3000, 8192, 16384])
def test_mass_gradient_with_a_gradient_on_p(nb, ctx, n):
    compare(nb, ctx, n, True, (128, 4, 128, 3, 1))


@pytest.mark.parametrize("n", [6000, 8192, 11000, 16384, 18000])
def test_mass_gradient_without_a_gradient_on_p(nb, ctx, n):
    compare(nb, ctx, n, False, (512, 2, 64, 1, 0))
