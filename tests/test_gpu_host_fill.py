"""Fills from host memory that only enqueue: the caller may be one fill ahead of
the GPU, and every fill sees its own hits, in place or copied, whatever was
staged before it."""
import numpy as np
import pytest

import oracle
from paper_1507_03074_gb300 import synth
from tests.test_gpu_parity import ht, _ob, _orr, random_hits  # noqa: F401

pytestmark = pytest.mark.gpu


def test_next_host_fill_is_staged_under_the_one_before(ht):
    """Two fills of a 4 GiB matrix (half a millisecond each): the second call
    returns while the first fill runs."""
    import torch
    b, r = ht.Binning(8, 32, 2048, 2048), ht.Ranges()
    ev = synth.make_event(*synth.split_hits(5000), seed=1)
    st = torch.cuda.Stream()
    ahead = 0
    with ht.Context(b, r, threshold=10, max_hits=5000) as ctx:
        for _ in range(6):
            end = torch.cuda.Event()
            ctx.fill(ev.x, ev.y, ev.z, stream=st)
            end.record(st)
            ctx.fill(ev.x, ev.y, ev.z, stream=st)
            ahead += not end.query()
            st.synchronize()
    assert ahead >= 3


def test_enqueued_host_fills_keep_their_hits(ht):
    """Fills of sizes around the one up to which hits are read in place (16384),
    back to back, each matrix against the oracle's."""
    import torch
    b, r = ht.Binning(2, 2, 40, 48), ht.Ranges()
    st = torch.cuda.Stream()
    sizes = (500, 16384, 1, 16385, 16384, 700, 0, 20000, 3, 16385, 16000, 16384)
    evs = [random_hits(n, 60 + i, rmax=900.0) for i, n in enumerate(sizes)]
    Ms = [torch.zeros(b.n_cells, dtype=torch.int32, device="cuda") for _ in sizes]
    torch.cuda.synchronize()
    with ht.Context(b, r, threshold=10, max_hits=20000) as ctx:
        for (x, y, z), M in zip(evs, Ms):
            a = [v.copy() for v in (x, y, z)]
            ctx.fill(*a, stream=st)
            for v in a:
                v.fill(np.nan)          # the caller may reuse its arrays at once
            ctx.matrix_into(M, stream=st)
        ctx.sync(stream=st)
    for (x, y, z), M in zip(evs, Ms):
        ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
        assert np.array_equal(M.cpu().numpy().view(np.uint32), ref.ravel())


@pytest.mark.parametrize("max_hits", [1, 2, 16383, 16384, 16385, 32768])
def test_host_staging_at_its_largest_fill(ht, max_hits):
    b, r = ht.Binning(1, 2, 20, 32), ht.Ranges()
    with ht.Context(b, r, threshold=10, max_hits=max_hits) as ctx:
        for k in range(4):
            x, y, z = random_hits(max_hits, 80 + k, rmax=900.0)
            ctx.fill(x, y, z)
            ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
            assert np.array_equal(ctx.matrix(), ref)
