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


KINDS = ["equal", "spectrum", "tracers", "span", "equal_si", "spectrum_si"]
BATCHES = {
    # every edge of a group, a tile and a block; empty clusters among them
    "edges": [1, 2, 31, 32, 33, 0, 63, 64, 65, 96, 127, 128, 129, 0, 191, 193, 255, 256, 257, 511, 513, 1000, 2049,
              4097, 4500, 1, 160],
    # blocks in several items, and one item per block
    "few": [1, 33, 65, 300],
    # several blocks per item
    "many": list(range(1, 4200, 37)) * 3,
}


def batch(sizes):
    """x, m, offsets, eps: the kinds of particles in turn."""
    parts = [particles(n, KINDS[i % len(KINDS)]) if n else (np.zeros((0, 3), "f4"), np.zeros(0, "f4"), np.float32(1))
             for i, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    return (np.concatenate([q[0] for q in parts]), np.concatenate([q[1] for q in parts]), off,
            np.array([q[2] for q in parts], np.float32))


def run_batch(nb, ctx, b, entry):
    """The plain or compensated force, or the compensated one on FP64 state."""
    import torch
    x, m, off, eps = (torch.from_numpy(v).cuda() for v in b)
    n = x.shape[0]
    a = torch.full((n, 3), float("nan"), device="cuda")
    p = torch.full((n,), float("nan"), device="cuda")
    if entry == 2:
        nb.nb_leapfrog_batched_step(ctx, x.double(), torch.zeros_like(x).double(), m, off, len(off) - 1, n, eps, a, p,
                                    0.0, 0, False, nb.NB_COMPENSATED)
    else:
        nb.nb_force_batched(ctx, x, m, off, len(off) - 1, n, eps, a, p, entry)
    nb.nb_synchronize(ctx)
    return a.cpu().numpy(), p.cpu().numpy()


@pytest.mark.parametrize("entry", [0, 1, 2])
@pytest.mark.parametrize("sizes", BATCHES)
def test_batched_edges_and_weights(nb, ctx, oracle_mod, sizes, entry):
    b = batch(BATCHES[sizes])
    a, p = run_batch(nb, ctx, b, entry)
    x, m, off, eps = b
    step = 7 if sizes == "many" else 1
    for c in range(0, len(off) - 1, step):
        lo, hi = off[c], off[c + 1]
        if hi > lo:
            ref = oracle_mod.force(x[lo:hi], m[lo:hi], eps[c])
            assert worst(a[lo:hi], p[lo:hi], *ref) <= TOL[min(entry, 1)], (c, hi - lo, KINDS[c % len(KINDS)])
    a2, p2 = run_batch(nb, ctx, b, entry)
    assert a.tobytes() == a2.tobytes() and p.tobytes() == p2.tobytes()


@pytest.mark.parametrize("entry", [0, 2])
def test_batched_bands(nb, ctx, entry):
    # A cluster whose blocks make more than one band, between two small ones:
    # rows of it against FP64 sums, with the measure and tolerance of the mode.
    sizes = [100, 100003, 64]
    b = batch(sizes)
    a, p = run_batch(nb, ctx, b, entry)
    x, m, off, eps = b
    lo, hi = off[1], off[2]
    X, M, e2 = x[lo:hi].astype(np.float64), m[lo:hi].astype(np.float64), float(eps[1]) ** 2
    rows = np.unique(np.concatenate([[0, sizes[1] - 1], workloads.sample_rows(sizes[1], 254, 4)]))
    for k in rows:
        d = X - X[k]
        y = 1 / np.sqrt((d * d).sum(1) + e2)
        y[k] = 0
        t = (M * y ** 3)[:, None] * d
        da = np.linalg.norm(a[lo + k].astype(np.float64) + t.sum(0))  # a is the sum over x_k - x_j
        assert da <= TOL[min(entry, 1)] * np.linalg.norm(t, axis=1).sum(), k
        assert abs(float(p[lo + k]) - M @ y) <= TOL[min(entry, 1)] * (M @ y), k


def test_batched_far_and_nonfinite_particles_as_the_direct_kernels(nb, ctx):
    sizes = [700, 1500, 90]
    x, m, off, eps = batch(sizes)
    for at in (off[0], off[1]):
        x[at + 7] = (3e19, 0, 0)
        x[at + 8] = (1e38, -1e38, 1e38)
        x[at + 400] = (np.inf, 0, 0)
        x[at + 640] = (0, np.nan, 0)
        m[at + 3] = np.inf
    for mode in (0, 1):
        a, p = run_batch(nb, ctx, (x, m, off, eps), mode)
        try:
            nb.nb_set_tile(ctx, mode, [t for t in nb.nb_list_tiles(mode) if not t.fused and not t.packed & 64][0])
            for c in range(len(sizes)):
                s = slice(off[c], off[c + 1])
                a0, p0 = run(nb, ctx, x[s], m[s], eps[c], mode)
                assert np.array_equal(np.isnan(a0), np.isnan(a[s])) and np.array_equal(np.isnan(p0), np.isnan(p[s]))
                assert np.array_equal(np.isinf(a0), np.isinf(a[s])) and np.array_equal(np.isinf(p0), np.isinf(p[s]))
        finally:
            nb.nb_set_tile(ctx, mode, None)


def test_batched_small_batch_after_a_large_one(nb, ctx):
    # The scratch holds the plan of another batch: results as on a fresh context.
    small = batch([5, 200, 77])
    with nb.Context(0) as fresh:
        want = run_batch(nb, fresh, small, 0)
    for sizes in (BATCHES["many"], [5, 200, 78], [200, 5, 77], [5, 200, 77]):
        got = run_batch(nb, ctx, batch(sizes), 0)
    assert got[0].tobytes() == want[0].tobytes() and got[1].tobytes() == want[1].tobytes()


@pytest.mark.parametrize("with_p", [False, True])
@pytest.mark.parametrize("n", [1, 33, 1000, 9728, 9729])
def test_plain_leapfrog_at_the_edge_of_the_single_launch_shapes(nb, ctx, n, with_p):
    # Three steps against the same steps with nb_force at the rounded positions: the
    # accelerations differ by at most 2e-5 of their scale (1e-5 each), so v by dt 3
    # times that and x by 3 dt times as much again; once up to 9728 (one kernel) by
    # the FP64 rounding alone. On a stream too, where the steps are replayed.
    import torch
    x32, m32, eps = particles(n, "spectrum")
    m = torch.from_numpy(m32).cuda()
    dt = 1.0 / 64
    x = torch.from_numpy(x32.astype(np.float64)).cuda() * (1 + 1e-9)
    v = torch.zeros_like(x)
    a, p = torch.empty((n, 3), device="cuda"), torch.empty(n, device="cuda")

    def force(x):
        nb.nb_force(ctx, x.float(), m, n, eps, a, p, 0)
        return a.double()

    wx, wv, g = x.clone(), v.clone(), force(x)
    for _ in range(3):
        wv -= 0.5 * dt * g
        wx += dt * wv
        g = force(wx)
        wv -= 0.5 * dt * g
    scale = float(g.abs().max())
    rel = 1e-14 if n <= 9728 else 2e-5
    nb.nb_synchronize(ctx)
    for stream in (None, torch.cuda.Stream()):
        gx, gv = x.clone(), v.clone()
        torch.cuda.synchronize()
        nb.nb_leapfrog_step(ctx, gx, gv, m, a, p if with_p else None, n, eps, dt, 3, 0, 0, stream)
        nb.nb_synchronize(ctx, stream)
        assert float((gv - wv).abs().max()) <= 3 * dt * rel * scale + 1e-15
        assert float((gx - wx).abs().max()) <= 9 * dt * dt * rel * scale + 1e-14


@pytest.mark.parametrize("first", [0, 1])
@pytest.mark.parametrize("n", [1, 33, 1000, 11000])
def test_adjoint_steps_in_the_vjp_kernels(nb, ctx, n, first):
    # The adjoint whose kicks and drift run in the mutual VJP's kernels against the
    # one with a direct VJP shape and kernels of their own: within the VJP's 1e-5.
    import torch
    x32, m32, eps = particles(n, "spectrum")
    rng = np.random.default_rng(n)
    m = torch.from_numpy(m32).cuda()
    x = torch.from_numpy(x32.astype(np.float64)).cuda()
    v, lx, lv, la = (torch.from_numpy(rng.normal(size=(n, 3))).cuda() for _ in range(4))
    lm = torch.from_numpy(rng.normal(size=n)).cuda()
    got = []
    try:
        for tile in (None, [t for t in nb.nb_list_vjp_tiles() if not t.packed & 64][0]):
            nb.nb_set_vjp_tile(ctx, tile)
            out = [t.clone() for t in (lx, lv, la, lm)]
            nb.nb_leapfrog_adjoint(ctx, x, v, None, m, n, eps, 1.0 / 64, 3, *out, first, 0)
            nb.nb_synchronize(ctx)
            got.append(out)
    finally:
        nb.nb_set_vjp_tile(ctx, None)
    for a, b in zip(*got):
        assert bool(torch.isfinite(a).all())
        assert float((a - b).norm()) <= 1e-5 * float(b.norm())
