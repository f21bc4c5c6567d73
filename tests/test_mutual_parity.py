"""GPU parity of the mutual pair kernels (each unordered pair evaluated once)
against the FP64 oracle, at the edges of their tiles, for every form of the
weights, and their bounded wait.

Tolerances are the modes' own (1e-5 plain, 1e-6 compensated; the measures of
test_force_parity.py): both modes run the same kernel, whose FP32 sums of at
most 256 terms enter compensated running sums, so its error stays near
sqrt(256) 2^-25 = 5e-7 at the worst particle.
"""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

TOL = {0: 1e-5, 1: 1e-6}


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


def mutual_tiles(nb, mode):
    return [t for t in nb.nb_list_tiles(mode) if t.packed & 64]


def run(nb, ctx, x32, m32, eps, mode):
    import torch
    n = x32.shape[0]
    xt, mt = torch.from_numpy(x32).cuda(), torch.from_numpy(m32).cuda()
    a = torch.full((n, 3), float("nan"), device="cuda")
    p = torch.full((n,), float("nan"), device="cuda")
    nb.nb_force(ctx, xt, mt, n, eps, a, p, mode)
    nb.nb_synchronize(ctx)
    return a.cpu().numpy(), p.cpu().numpy()


def worst(a, p, ra, rp, ramag):
    da = np.linalg.norm(a.astype(np.float64) - ra, axis=1)
    dp = np.abs(p.astype(np.float64) - rp)
    ea = np.where(ramag > 0, da / np.where(ramag > 0, ramag, 1.0), da)
    ep = np.where(rp > 0, dp / np.where(rp > 0, rp, 1.0), dp)
    return max(ea.max(), ep.max())


def particles(n, kind):
    """x, m, eps of a Plummer sphere: equal masses; a spectrum over a factor of
    30; a spectrum with massless tracers; masses over a factor of 2^40; and
    equal or unequal masses in units of kilograms and metres."""
    x, _, m = workloads.plummer(n, seed=n + len(kind))
    rng = np.random.default_rng(n)
    eps = 1.0 / 64
    if kind != "equal" and kind != "equal_si":
        m = m * np.exp(rng.uniform(0, np.log(30), n))
    if kind == "tracers":
        m[rng.random(n) < 0.3] = 0.0
    if kind == "span":
        m = m * 2.0 ** rng.integers(-20, 21, n)
    if kind.endswith("_si"):
        x, m, eps = x * 3.1e16, m * 2e33, eps * 3.1e16
    return x.astype(np.float32), m.astype(np.float32), np.float32(eps)


@pytest.mark.parametrize("kind", ["equal", "spectrum", "tracers", "span", "equal_si", "spectrum_si"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 129, 1023, 1024, 1025, 2500, 4100])
def test_tile_edges_and_weights(nb, ctx, oracle_mod, n, kind):
    x32, m32, eps = particles(n, kind)
    ra, rp, ramag = oracle_mod.force(x32, m32, eps)
    for mode in (0, 1):
        try:
            for tile in mutual_tiles(nb, mode):
                nb.nb_set_tile(ctx, mode, tile)
                a, p = run(nb, ctx, x32, m32, eps, mode)
                assert worst(a, p, ra, rp, ramag) <= TOL[mode], (tile, mode)
                a2, p2 = run(nb, ctx, x32, m32, eps, mode)
                assert a.tobytes() == a2.tobytes() and p.tobytes() == p2.tobytes(), tile
        finally:
            nb.nb_set_tile(ctx, mode, None)


def test_far_and_nonfinite_particles_as_the_direct_kernels(nb, ctx):
    # Coordinates whose squared distances overflow FP32, infinities and NaN:
    # finite, infinite and NaN results in the same places as the direct kernels'.
    x32, m32, eps = particles(1500, "spectrum")
    x32[7] = (3e19, 0, 0)
    x32[8] = (1e38, -1e38, 1e38)
    x32[900] = (np.inf, 0, 0)
    x32[1400] = (0, np.nan, 0)
    m32[3] = np.inf
    for mode in (0, 1):
        try:
            nb.nb_set_tile(ctx, mode, [t for t in nb.nb_list_tiles(mode) if not t.fused and not t.packed & 64][0])
            a0, p0 = run(nb, ctx, x32, m32, eps, mode)
            for tile in mutual_tiles(nb, mode):
                nb.nb_set_tile(ctx, mode, tile)
                a1, p1 = run(nb, ctx, x32, m32, eps, mode)
                assert np.array_equal(np.isnan(a0), np.isnan(a1)) and np.array_equal(np.isnan(p0), np.isnan(p1))
                assert np.array_equal(np.isinf(a0), np.isinf(a1)) and np.array_equal(np.isinf(p0), np.isinf(p1))
        finally:
            nb.nb_set_tile(ctx, mode, None)


def test_bounded_wait_reports_timeout_and_context_survives(nb, ctx, oracle_mod):
    # One tile's copy is never issued: the CTA's bounded wait (0.2 s) runs out,
    # nb_synchronize reports it, and the next call is correct.
    x32, m32, eps = particles(3000, "spectrum")
    nb.nb_set_tile(ctx, 0, mutual_tiles(nb, 0)[0])
    try:
        nb.nb_debug_set_fault(ctx, 3, 200_000_000)
        try:
            with pytest.raises(nb.NBError) as e:
                run(nb, ctx, x32, m32, eps, 0)
            assert e.value.status == nb.NB_ERR_TIMEOUT
        finally:
            nb.nb_debug_set_fault(ctx, -1, 0)
        a, p = run(nb, ctx, x32, m32, eps, 0)
    finally:
        nb.nb_set_tile(ctx, 0, None)
    assert worst(a, p, *oracle_mod.force(x32, m32, eps)) <= TOL[0]


@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 511, 512, 513, 1025, 2100])
def test_vjp_tile_edges(nb, ctx, oracle_mod, n):
    # The adjoint's mutual shapes at the edges of their tiles, with and without
    # an upstream gradient on p, masses of both signs and zero among them: the
    # measure and tolerance of test_vjp_parity.py.
    import torch
    from test_vjp_parity import rel_to_scale, vjp_term_scales
    x32, m32, eps = particles(n, "tracers")
    m32[::3] *= -1
    rng = np.random.default_rng(n)
    ga = rng.normal(size=(n, 3)).astype(np.float32)
    gp = rng.normal(size=n).astype(np.float32)
    dev = [torch.from_numpy(v).cuda() for v in (x32, m32, ga, gp)]
    try:
        for tile in [t for t in nb.nb_list_vjp_tiles() if t.packed & 64]:
            nb.nb_set_vjp_tile(ctx, tile)
            for with_gp in (True, False):
                gx = torch.full((n, 3), float("nan"), device="cuda")
                gm = torch.full((n,), float("nan"), device="cuda")
                nb.nb_force_vjp(ctx, dev[0], dev[1], n, eps, dev[2], dev[3] if with_gp else None, gx, gm)
                nb.nb_synchronize(ctx)
                g0 = gp if with_gp else np.zeros_like(gp)
                rgx, rgm = oracle_mod.force_vjp(x32, m32, eps, ga, g0)
                sx, sm = vjp_term_scales(x32, np.abs(m32), eps, ga, g0)
                one = np.finfo(np.float32).tiny
                assert rel_to_scale(gx.cpu().numpy(), rgx, sx + one) <= 1e-5, (tile, with_gp)
                assert rel_to_scale(gm.cpu().numpy(), rgm, sm + one) <= 1e-5, (tile, with_gp)
    finally:
        nb.nb_set_vjp_tile(ctx, None)


def test_vjp_panels(nb, ctx):
    # 200000 particles: the j-side sums exceed the bound on the scratch, so the
    # rows run in panels. 128 particles, the first and last among them, against
    # FP64 rows of the formulas in test_vjp_parity.py, with that file's measure
    # and tolerance.
    import torch
    n = 200000
    x32, m32, eps = particles(n, "spectrum")
    rng = np.random.default_rng(3)
    ga = rng.normal(size=(n, 3)).astype(np.float32)
    gp = rng.normal(size=n).astype(np.float32)
    x, m, gat, gpt = (torch.from_numpy(v).cuda() for v in (x32, m32, ga, gp))
    gx, gm = torch.empty((n, 3), device="cuda"), torch.empty(n, device="cuda")
    try:
        nb.nb_set_vjp_tile(ctx, [t for t in nb.nb_list_vjp_tiles() if t.packed & 64][-1])
        nb.nb_force_vjp(ctx, x, m, n, eps, gat, gpt, gx, gm)
        nb.nb_synchronize(ctx)
    finally:
        nb.nb_set_vjp_tile(ctx, None)
    rows = np.unique(np.concatenate([[0, n - 1], workloads.sample_rows(n, 126, 4)]))
    for k in rows:
        X, M, GA, GP = x32.astype(np.float64), m32.astype(np.float64), ga.astype(np.float64), gp.astype(np.float64)
        r = X[k] - X
        r2 = (r * r).sum(1)
        y = 1 / np.sqrt(r2 + float(eps) ** 2)
        y[k] = 0
        rk, rl, rn = r @ GA[k], (r * GA).sum(1), np.sqrt(r2)
        c = 3 * y ** 5 * (M[k] * rl - M * rk) - y ** 3 * (GP[k] * M + M[k] * GP)
        want_x = c @ r + GA[k] * (M @ y ** 3) - M[k] * (y ** 3 @ GA)
        want_m = GP @ y - rl @ y ** 3
        na = np.linalg.norm(GA, axis=1)
        sx = (M * (y ** 3 * na[k] + 3 * y ** 5 * abs(rk) * rn + abs(GP[k]) * y ** 3 * rn)
              + M[k] * (y ** 3 * na + 3 * y ** 5 * abs(rl) * rn + abs(GP) * y ** 3 * rn)).sum()
        sm = (abs(rl) * y ** 3 + abs(GP) * y).sum()
        assert np.linalg.norm(gx[k].cpu().numpy() - want_x) <= 1e-5 * sx, k
        assert abs(float(gm[k]) - want_m) <= 1e-5 * sm, k
