"""GPU: the mutual force kernels where the j-side sums exceed the scratch set aside and
the rows run in several panels (above about 370000 FP32 particles, 320000 on two-word
positions): rows of particles, the first and last among them, against FP64 sums, with the
modes' own tolerances and the measure of test_force_parity.py."""
import numpy as np
import pytest

import workloads
from test_mutual_parity import TOL, ctx, nb, particles  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu

N = 400003


def check(a, p, x, m, eps, tol):
    import torch
    rows = np.unique(np.concatenate([[0, N - 1], workloads.sample_rows(N, 126, 4)]))
    m = m.double()
    for k in range(0, len(rows), 32):
        r = torch.from_numpy(rows[k:k + 32]).cuda()
        d = x[r][:, None] - x[None]
        y = (d.square().sum(-1) + float(eps) ** 2).rsqrt()
        y[torch.arange(len(r)), r] = 0
        t = (m * y ** 3)[..., None] * d
        want_p = (m * y).sum(1)
        assert ((a[r].double() - t.sum(1)).norm(dim=1) <= tol * t.norm(dim=2).sum(1)).all()
        assert ((p[r].double() - want_p).abs() <= tol * want_p).all()


@pytest.mark.parametrize("kind", ["equal", "spectrum", "tracers"])
@pytest.mark.parametrize("entry", ["force", "state"])
def test_rows_of_several_panels(nb, ctx, entry, kind):
    import torch
    x32, m32, eps = particles(N, kind)
    m = torch.from_numpy(m32).cuda()
    a, p = torch.full((N, 3), float("nan"), device="cuda"), torch.full((N,), float("nan"), device="cuda")
    if entry == "force":
        x = torch.from_numpy(x32).cuda()
        nb.nb_force(ctx, x, m, N, eps, a, p, nb.NB_COMPENSATED)
    else:
        x = torch.from_numpy(x32.astype(np.float64)).cuda() * (1 + 1e-9)
        nb.nb_leapfrog_step(ctx, x, torch.zeros_like(x), m, a, p, N, eps, 0.0, 0, False, nb.NB_COMPENSATED)
    nb.nb_synchronize(ctx)
    check(a, p, x.double(), m, eps, TOL[1])
