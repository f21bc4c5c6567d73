"""GPU: the compensated force of FP64 state is no less exact than with the direct kernel
that summed 128 j-particles at a time (which no longer runs where the mutual kernels'
scratch can be had): its errors on the same systems, measured on a GB300, are the bounds.
2-norms over 2048 particles against FP64, root mean squares over six Plummer spheres; 2%
for chance."""
import numpy as np
import pytest

import workloads
from test_mutual_parity import ctx, nb  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,direct_a,direct_p", [(12000, 4.96e-8, 2.95e-8), (20000, 4.37e-8, 2.74e-8)])
def test_compensated_state(nb, ctx, n, direct_a, direct_p):
    import torch
    eps, rows = 1.0 / 64, np.sort(np.random.default_rng(1).choice(n, 2048, replace=False))
    ea, ep = [], []
    for seed in range(6):
        x, v, m = workloads.plummer(n, seed=n + 1000 * seed)
        x, v, m = torch.from_numpy(x).cuda(), torch.from_numpy(v).cuda(), torch.from_numpy(m.astype(np.float32)).cuda()
        a, p = torch.empty((n, 3), device="cuda"), torch.empty(n, device="cuda")
        nb.nb_leapfrog_step(ctx, x, v, m, a, p, n, eps, 0.0, 0, False, nb.NB_COMPENSATED)
        nb.nb_synchronize(ctx)
        want_a, want_p = [], []
        for k in range(0, len(rows), 64):
            r = torch.from_numpy(rows[k:k + 64]).cuda()
            d = x[r][:, None] - x[None]
            y = (d.square().sum(-1) + eps ** 2).rsqrt()
            y[torch.arange(len(r)), r] = 0
            want_a.append(((m.double() * y ** 3)[..., None] * d).sum(1))
            want_p.append((m.double() * y).sum(1))
        r, want_a, want_p = torch.from_numpy(rows).cuda(), torch.cat(want_a), torch.cat(want_p)
        ea.append(float((a[r].double() - want_a).norm() / want_a.norm()))
        ep.append(float((p[r].double() - want_p).norm() / want_p.norm()))
    assert np.sqrt(np.mean(np.square(ea))) <= 1.02 * direct_a
    assert np.sqrt(np.mean(np.square(ep))) <= 1.02 * direct_p
