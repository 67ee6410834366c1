"""The per-kernel profile names every kernel kind, the last ones too."""
import numpy as np
import pytest

from tests.test_gpu_parity import ht, random_hits  # noqa: F401

pytestmark = pytest.mark.gpu


def test_profile_holds_every_kernel(ht):
    import torch
    b = ht.Binning(1, 2, 64, 64)
    x, y, z = random_hits(300, 3)
    M = torch.zeros(b.n_cells, dtype=torch.int32, device="cuda")
    with ht.Context(b, ht.Ranges(), threshold=4, max_hits=600) as ctx:
        ctx.profile(True)
        before = ctx.launches
        ctx.fill(x, y, z)
        ctx.fill(x[:2], y[:2], z[:2], accumulate=True)
        ctx.matrix_into(M)
        ctx.find_maxima(capacity=64)
        prof = ctx.profile_read()
        assert prof["k_copy"][0] == 1
        assert sum(n for n, _ in prof.values()) == ctx.launches - before
    with ht.Batch(b, ht.Ranges(), threshold=4, max_events=1, max_hits=600, capacity=64) as B:
        B.profile(True)
        B.run(*ht.Batch.concat([(x, y, z)]))
        batch = B.profile_read()
        assert batch.keys() == prof.keys() and batch["k_fill_tma"][0] == 1 and batch["k_copy"][0] == 0
        assert all(np.isfinite(t) for _, t in batch.values())
