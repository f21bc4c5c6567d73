"""GPU: a captured nb_force keeps its scratch while other calls of the context take
theirs (the header's promise on graph capture)."""
import numpy as np
import pytest

import workloads
from test_mutual_parity import ctx, nb  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1])
def test_replay_after_calls_with_larger_scratch(nb, mode):
    # 25000 particles take a mutual shape in both modes. The calls in between need more
    # of every kind of scratch than nb_force: two records per particle, twice the sums,
    # more particles.
    import torch
    n, eps = 25000, 1.0 / 64
    x64, v, m = workloads.plummer(n, seed=1)
    x, mt = torch.from_numpy(x64.astype(np.float32)).cuda(), torch.from_numpy(m.astype(np.float32)).cuda()
    a, p = torch.empty((n, 3), device="cuda"), torch.empty(n, device="cuda")
    with nb.Context(0) as ctx:
        nb.nb_reserve(ctx, n, mode)
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            nb.nb_force(ctx, x, mt, n, eps, a, p, mode, side)
        side.synchronize()
        want = a.cpu(), p.cpu()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            nb.nb_force(ctx, x, mt, n, eps, a, p, mode)

        gx, gm, b, q = torch.empty_like(a), torch.empty_like(p), torch.empty_like(a), torch.empty_like(p)
        nb.nb_force_vjp(ctx, x, mt, n, eps, x, p, gx, gm)
        x2, v2 = torch.from_numpy(x64.copy()).cuda(), torch.from_numpy(v.copy()).cuda()
        nb.nb_leapfrog_step(ctx, x2, v2, mt, b, q, n, eps, 1e-3, 3, False, nb.NB_COMPENSATED)
        nb.nb_energy(ctx, x2, v2, mt, n, eps, nb.NB_COMPENSATED)
        big = 4 * n
        xb, mb = x.repeat(4, 1), mt.repeat(4)
        ab, pb = torch.empty((big, 3), device="cuda"), torch.empty(big, device="cuda")
        off = torch.tensor([0, big], device="cuda")
        nb.nb_force_batched(ctx, xb, mb, off, 1, big, torch.tensor([eps], device="cuda"), ab, pb, mode)
        nb.nb_synchronize(ctx)

        a.fill_(float("nan"))
        p.fill_(float("nan"))
        graph.replay()
        nb.nb_synchronize(ctx)
        assert torch.equal(a.cpu(), want[0]) and torch.equal(p.cpu(), want[1])


def test_reserved_scratch_serves_smaller_calls(nb):
    # 371000 particles run in two panels of rows, 370000 in one that has more rows than
    # either: after nb_reserve for the former, the latter allocates nothing.
    import torch
    n, small = 371000, 370000
    x = torch.randn(n, 3, device="cuda")
    m, a, p = torch.ones(n, device="cuda"), torch.empty((n, 3), device="cuda"), torch.empty(n, device="cuda")
    with nb.Context(0) as ctx:
        nb.nb_reserve(ctx, n, 0)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):  # an allocation here is an error
            nb.nb_force(ctx, x, m, small, 0.01, a, p, 0)
        graph.replay()
        nb.nb_synchronize(ctx)
        assert torch.isfinite(a[:small]).all() and torch.isfinite(p[:small]).all()
