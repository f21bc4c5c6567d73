"""GPU: ranges of the mutual kernels' weights for unequal masses. Softening lengths
from 2^-39 to 2^39, masses spread over a factor of 2^10 or 2^27 with the first
particle the lightest or the heaviest, in units of one or (from eps = 1 on) of
2^80, against the FP64 oracle: nb_force on every mutual shape, the compensated
force of FP64 state, and a batch. Every result is far inside FP32's range, so the
modes' own tolerances hold (1e-5 plain, 1e-6 compensated; test_mutual_parity.py has
the measures and the reason)."""
import numpy as np
import pytest

import workloads
from test_mutual_parity import TOL, ctx, mutual_tiles, nb, run, run_batch, worst  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu

CASES = [(e, spread, first, unit) for e in range(-39, 40, 6) for spread in (10, 27) for first in ("lightest", "heaviest")
         for unit in ((0, 80) if e > 0 else (0,))]


def system(n, e, spread, first, unit):
    x, _, _ = workloads.plummer(n, seed=n)
    eps = np.float32(1.3 * 2.0 ** e)
    rng = np.random.default_rng(n + spread)
    m = 1.7 * 2.0 ** (unit + rng.uniform(0, spread, n))
    k = m.argmin() if first == "lightest" else m.argmax()
    m[[0, k]] = m[[k, 0]]
    return (x * min(64 * float(eps), 2.0 ** 32)).astype(np.float32), m.astype(np.float32), eps


@pytest.mark.parametrize("e,spread,first,unit", CASES)
def test_force_at_every_scale(nb, ctx, oracle_mod, e, spread, first, unit):
    x, m, eps = system(1500, e, spread, first, unit)
    ref = oracle_mod.force(x, m, eps)
    try:
        for tile in mutual_tiles(nb, 0):
            nb.nb_set_tile(ctx, 0, tile)
            assert worst(*run(nb, ctx, x, m, eps, 0), *ref) <= TOL[0], tile
    finally:
        nb.nb_set_tile(ctx, 0, None)


@pytest.mark.parametrize("e,spread,first,unit", CASES)
def test_compensated_state_at_every_scale(nb, ctx, oracle_mod, e, spread, first, unit):
    import torch
    x, m, eps = system(1100, e, spread, first, unit)
    xt, mt = torch.from_numpy(x.astype(np.float64)).cuda(), torch.from_numpy(m).cuda()
    a, p = torch.empty((len(m), 3), device="cuda"), torch.empty(len(m), device="cuda")
    nb.nb_leapfrog_step(ctx, xt, torch.zeros_like(xt), mt, a, p, len(m), eps, 0.0, 0, False, nb.NB_COMPENSATED)
    nb.nb_synchronize(ctx)
    assert worst(a.cpu().numpy(), p.cpu().numpy(), *oracle_mod.force(x, m, eps)) <= TOL[1]


@pytest.mark.parametrize("entry", [0, 2])
def test_batch_of_every_scale(nb, ctx, oracle_mod, entry):
    parts = [system(300 + 17 * k, *c) for k, c in enumerate(CASES)]
    off = np.concatenate([[0], np.cumsum([len(q[1]) for q in parts])]).astype(np.int64)
    b = (np.concatenate([q[0] for q in parts]), np.concatenate([q[1] for q in parts]), off,
         np.array([q[2] for q in parts], np.float32))
    a, p = run_batch(nb, ctx, b, entry)
    for k, (x, m, eps) in enumerate(parts):
        lo, hi = off[k], off[k + 1]
        assert worst(a[lo:hi], p[lo:hi], *oracle_mod.force(x, m, eps)) <= TOL[min(entry, 1)], CASES[k]
