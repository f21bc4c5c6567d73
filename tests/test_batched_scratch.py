"""GPU: the scratch that a batch of many small clusters leaves in its context."""
import pytest

from test_mutual_parity import nb  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


def test_many_small_clusters_take_what_their_blocks_need(nb):
    # 100000 clusters of 64: 150000 padded blocks of 4.1 KiB, 52 MiB of items' sums and
    # at most 512 MiB of j-side sums, which clusters of up to 256 do not have.
    import torch
    c, size = 100000, 64
    n = c * size
    x, m = torch.randn(n, 3, device="cuda"), torch.full((n,), 1.0 / size, device="cuda")
    off = torch.arange(c + 1, device="cuda") * size
    eps, a, p = torch.full((c,), 0.05, device="cuda"), torch.empty(n, 3, device="cuda"), torch.empty(n, device="cuda")
    with nb.Context(0) as ctx:
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        nb.nb_force_batched(ctx, x, m, off, c, n, eps, a, p, 0)
        nb.nb_synchronize(ctx)
        used = free - torch.cuda.mem_get_info()[0]
        assert used <= 150000 * 4300 + (600 << 20), used
        assert torch.isfinite(a).all() and torch.isfinite(p).all()
