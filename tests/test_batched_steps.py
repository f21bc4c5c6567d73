"""GPU: several steps of the batched leap-frog in one call (one plan, the queue and the
forms of the weights handed on from step to step, replayed from a graph on a side
stream) give the bits of as many calls of one step."""
import numpy as np
import pytest

from test_mutual_parity import BATCHES, batch, ctx, nb  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side_stream", [False, True])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("sizes", ["edges", "few"])
def test_steps_in_one_call_and_apart(nb, ctx, sizes, mode, side_stream):
    import torch
    x32, m32, off, eps = batch(BATCHES[sizes])
    m, off, eps = (torch.from_numpy(v).cuda() for v in (m32, off, eps))
    n, c, dt = len(m32), len(off) - 1, 2.0 ** -20
    stream = torch.cuda.Stream() if side_stream else None
    got = []
    for calls, steps in ((1, 5), (5, 1)):
        x = torch.from_numpy(x32.astype(np.float64)).cuda()
        v = x * 0.25
        a, p = torch.empty((n, 3), device="cuda"), torch.empty(n, device="cuda")
        torch.cuda.synchronize()
        for k in range(calls):
            nb.nb_leapfrog_batched_step(ctx, x, v, m, off, c, n, eps, a, p, dt, steps, k > 0, mode, stream)
        nb.nb_synchronize(ctx, stream)
        got.append([t.cpu().numpy().tobytes() for t in (x, v, a, p)])
    assert got[0] == got[1]
