"""GPU: nb_energy's potential kernels (no accelerations) sum what the packed
shapes of nb_force sum: the same bits of p, so the same W to the FP64 rounding
of its sum over particles, at one size of each built-in shape and at the edges
of their tiles; and the compensated mode against FP64."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

# nb_tile of the built-in packed shape per size class (threads, ipt, jtile, stages, unroll, minblocks, release)
SMALL, MID, LARGE, HUGE = ((256, 2, 128, 4, 4, 1, 0), (64, 4, 128, 4, 4, 1, 0), (256, 4, 512, 3, 4, 1, 0),
                           (256, 4, 1024, 3, 4, 1, 0))
SHAPES = {1: SMALL, 1025: SMALL, 8191: SMALL, 8192: MID, 20011: MID, 32768: LARGE, 40001: LARGE, 131072: HUGE,
          140007: HUGE}


@pytest.fixture(scope="module")
def nb():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0904_3659_gb300 import build
    build.build()
    import paper_0904_3659_gb300 as nbmod
    return nbmod


@pytest.fixture(scope="module")
def ctx(nb):
    c = nb.Context(0)
    yield c
    c.close()


def system(n):
    import torch
    x, v, m = workloads.plummer(n, seed=n)
    m = m * np.exp(np.random.default_rng(n).uniform(0, np.log(30), n))
    return (torch.from_numpy(x.astype(np.float32)).cuda(), torch.from_numpy(v).cuda(),
            torch.from_numpy(m.astype(np.float32)).cuda())


@pytest.mark.parametrize("n", SHAPES)
def test_plain_potential_is_the_packed_shapes(nb, ctx, n):
    import torch
    x, v, m = system(n)
    a, p = torch.empty_like(x), torch.empty_like(m)
    _, w = nb.nb_energy(ctx, x.double(), v, m, n, 1 / 64, 0)
    try:
        nb.nb_set_tile(ctx, 0, [t for t in nb.nb_list_tiles(0) if not t.fused and not t.packed & 64
                                and (t.threads, t.ipt, t.jtile, t.stages, t.unroll, t.minblocks, t.release) == SHAPES[n]
                                and t.packed & 63 == 63 and t.refine == 0 and t.sums_in_smem == 0][0])
        nb.nb_force(ctx, x, m, n, 1 / 64, a, p, 0)
        nb.nb_synchronize(ctx)
    finally:
        nb.nb_set_tile(ctx, 0, None)
    want = float((-0.5 * m.double() * p.double()).sum())
    assert abs(w - want) <= 1e-13 * abs(want)


@pytest.mark.parametrize("n", [1, 255, 1025, 20011, 40001])
def test_compensated_potential_against_fp64(nb, ctx, n):
    # p within 1e-6 per particle, so W (all terms of one sign) too.
    import torch
    x, v, m = system(n)
    _, w = nb.nb_energy(ctx, x.double(), v, m, n, 1 / 64, 1)
    X, M, want = x.double(), m.double(), 0.0
    for k in range(0, n, 2048):
        y = ((X[k:k + 2048, None] - X[None]).square().sum(-1) + (1 / 64) ** 2).rsqrt()
        y[torch.arange(y.shape[0]), torch.arange(k, k + y.shape[0])] = 0
        want -= 0.5 * float((M[k:k + 2048] * (y @ M)).sum())
    assert abs(w - want) <= 1e-6 * abs(want)
