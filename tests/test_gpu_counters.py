"""What a tile fill and its ordering leave in the counters: a scan that no
binning precedes -- one behind a captured scan, the autotuner's fills -- starts
from zero."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_parity import ht, _ob, _orr, assert_peaks_equal, random_hits  # noqa: F401

pytestmark = pytest.mark.gpu


def test_scan_behind_a_captured_scan(ht):
    """The captured scan does not run when it is captured, so the one after it
    cannot rely on anything that it would clear."""
    import torch
    b, r, T = ht.Binning(2, 3, 50, 64), ht.Ranges(), 3
    x, y, z = random_hits(900, 4)
    M_ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
    pk_ref, n_ref = oracle.find_maxima(_ob(b), _orr(r), M_ref, T)
    st = torch.cuda.Stream()
    out = torch.zeros(n_ref, 8, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    with ht.Context(b, r, threshold=T, max_hits=x.size) as ctx:
        ctx.fill(x, y, z, stream=st)
        ctx.find_maxima(capacity=n_ref, out=out, count=cnt, stream=st)   # orders the tile fill's peaks
        ctx.sync(stream=st)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            ctx.find_maxima(capacity=n_ref, out=out, count=cnt, stream=st)
        for run in ("eager", "replay", "eager"):
            out.zero_()
            cnt.zero_()
            torch.cuda.synchronize()
            if run == "eager":
                ctx.find_maxima(capacity=n_ref, out=out, count=cnt, stream=st)
            else:
                with torch.cuda.stream(st):
                    g.replay()
            ctx.sync(stream=st)
            assert int(cnt.item()) == n_ref, run
            assert_peaks_equal(out.cpu().numpy().view(ht.PEAK_DTYPE).reshape(-1), pk_ref)


@pytest.mark.parametrize("find_first", [True, False])
def test_autotune_behind_a_dense_tile_fill(ht, find_first):
    """Nearly every vote falls into a cell of its own, and every cell is a
    candidate: the peaks of the tile fill and the candidates of another fill
    together are more than the entries hold."""
    b, r, T, n = ht.Binning(1, 1, 64, 4096), ht.Ranges(), 1, 256
    rng = np.random.default_rng(5)
    rad, ph = rng.uniform(30, 500, n), rng.uniform(0.35, 1.2, n) * rng.choice([-1, 1], n)
    x, y, z = (a.astype(np.float32) for a in (rad * np.sin(ph), rad * np.cos(ph), rng.uniform(-300, 300, n)))
    M_ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
    pk_ref, n_ref = oracle.find_maxima(_ob(b), _orr(r), M_ref, T)
    assert n_ref + int((M_ref > 0).sum()) > n * b.n_a + 1 + 2048
    with ht.Context(b, r, threshold=T, max_hits=n) as ctx:
        ctx.fill(x, y, z)
        if find_first:
            pk, total = ctx.find_maxima(capacity=1 << 15)
            assert total == n_ref
        ctx.autotune(reps=1)
        for _ in range(2):
            pk, total = ctx.find_maxima(capacity=1 << 15)
            assert total == n_ref
            assert_peaks_equal(pk, pk_ref)
        assert np.array_equal(ctx.matrix(), M_ref)
