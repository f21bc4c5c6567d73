"""GPU: the VJP's mutual shapes in units of metres and kilograms, where a mass times a
distance leaves FP32's range but no result does: against the oracle, with the measure
and tolerance of test_vjp_parity.py."""
import numpy as np
import pytest

import workloads
from test_mutual_parity import ctx, nb  # noqa: F401 (fixtures)
from test_vjp_parity import rel_to_scale, vjp_term_scales

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mass,length,eps", [(2e30, 1e11, 1e8), (1e30, 1e9, 1e7), (6e24, 1e12, 1e10)])
@pytest.mark.parametrize("n", [33, 1100])
def test_metres_and_kilograms(nb, ctx, oracle_mod, n, mass, length, eps):
    import torch
    x, _, _ = workloads.plummer(n, seed=n)
    rng = np.random.default_rng(n)
    x32 = (x * length).astype(np.float32)
    m32 = (mass * np.exp(rng.uniform(0, np.log(30), n))).astype(np.float32)
    ga, gp = rng.normal(size=(n, 3)).astype(np.float32), rng.normal(size=n).astype(np.float32)
    eps = np.float32(eps)
    want_x, want_m = oracle_mod.force_vjp(x32, m32, eps, ga, gp)
    sx, sm = vjp_term_scales(x32, m32, eps, ga, gp)
    dev = [torch.from_numpy(v).cuda() for v in (x32, m32, ga, gp)]
    try:
        for tile in [t for t in nb.nb_list_vjp_tiles() if t.packed & 64]:
            nb.nb_set_vjp_tile(ctx, tile)
            gx, gm = torch.empty_like(dev[0]), torch.empty_like(dev[1])
            nb.nb_force_vjp(ctx, dev[0], dev[1], n, eps, dev[2], dev[3], gx, gm)
            nb.nb_synchronize(ctx)
            assert rel_to_scale(gx.cpu().numpy(), want_x, sx) <= 1e-5, tile
            assert rel_to_scale(gm.cpu().numpy(), want_m, sm) <= 1e-5, tile
    finally:
        nb.nb_set_vjp_tile(ctx, None)
