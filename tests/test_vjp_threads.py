"""GPU: contexts of several threads run the VJP side by side at sizes whose launches ask
for different amounts of shared memory (a limit that belongs to the kernel, not to the
context): every call succeeds with the bits of a call alone."""
import threading

import numpy as np
import pytest

import workloads
from test_mutual_parity import nb  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


def test_contexts_of_several_threads(nb):
    import torch
    sizes, eps, errors = (300, 1000, 4096, 5000), 1.0 / 64, []
    data, want = {}, {}
    for n in sizes:
        x, _, m = workloads.plummer(n, seed=n)
        ga = np.random.default_rng(n).normal(size=(n, 3))
        data[n] = [torch.from_numpy(v.astype(np.float32)).cuda() for v in (x, m, ga, ga[:, 0].copy())]

    def call(ctx, n, stream):
        x, m, ga, gp = data[n]
        with torch.cuda.stream(stream):
            gx, gm = torch.empty_like(x), torch.empty_like(m)
        nb.nb_force_vjp(ctx, x, m, n, eps, ga, gp, gx, gm, stream)
        nb.nb_synchronize(ctx, stream)
        return gx, gm

    with nb.Context(0) as ctx:
        for n in sizes:
            want[n] = call(ctx, n, torch.cuda.Stream())
    torch.cuda.synchronize()

    def work(mine):
        try:
            stream = torch.cuda.Stream()
            for _ in range(4):
                with nb.Context(0) as ctx:
                    for k in range(20):
                        n = sizes[(k + mine) % len(sizes)]
                        got = call(ctx, n, stream)
                        if not (torch.equal(got[0], want[n][0]) and torch.equal(got[1], want[n][1])):
                            errors.append((mine, n))
        except Exception as e:  # reported by the test's thread
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:5]
