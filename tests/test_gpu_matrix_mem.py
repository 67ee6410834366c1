"""The vote matrices' memory on both sides of the size from which it is
compressible: the contents are the oracle's through fills, copies out and in,
the paper's fill and accumulation, and destroying a context gives its memory
back."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_parity import ht, _ob, _orr, assert_peaks_equal, random_hits  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_a", [2047, 2048, 4096], ids=["below_32MiB", "32MiB", "64MiB"])
def test_matrix_memory_holds_the_counts(ht, n_a):
    b, r, T = ht.Binning(1, 2, n_a, 2048), ht.Ranges(), 3
    x, y, z = random_hits(600, n_a)
    M_ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
    pk_ref, n_ref = oracle.find_maxima(_ob(b), _orr(r), M_ref, T)
    with ht.Context(b, r, threshold=T, max_hits=1200) as ctx:
        for fills in (((0, 600, {}),), ((0, 600, dict(naive=True)),), ((0, 200, {}), (200, 600, dict(accumulate=True)))):
            for i, j, kw in fills:
                ctx.fill(x[i:j], y[i:j], z[i:j], **kw)
            pk, n = ctx.find_maxima(capacity=1 << 16)
            assert n == n_ref
            assert_peaks_equal(pk, pk_ref)
            assert np.array_equal(ctx.matrix(), M_ref)
        noise = np.random.default_rng(1).integers(0, 1 << 32, M_ref.shape, dtype=np.uint32)
        ctx.set_matrix(noise)
        assert np.array_equal(ctx.matrix(), noise)


def test_matrix_memory_is_given_back(ht):
    import torch
    b, r = ht.Binning(4, 16, 512, 1024), ht.Ranges()   # 128 MiB
    ctx = ht.Context(b, r, threshold=3, max_hits=16)
    ctx.close()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(5):
        ctxs = [ht.Context(b, r, threshold=3, max_hits=16) for _ in range(3)]
        assert torch.cuda.mem_get_info()[0] <= free - 3 * b.n_cells * 4
        for c in ctxs:
            c.close()
    assert torch.cuda.mem_get_info()[0] >= free - (8 << 20)


@pytest.mark.parametrize("bins", [(1, 1, 1, 3), (1, 1, 2, 4), (1, 2, 31, 33), (2, 3, 64, 128), (1, 5, 1023, 9)], ids=str)
@pytest.mark.parametrize("shift", [0, 1, 4, 8])
def test_matrix_into_device_memory(ht, bins, shift):
    """The matrix copied to device memory at any word, to its last cell and
    not beyond."""
    import torch
    b, n = ht.Binning(*bins), 300
    x, y, z = random_hits(n, 9, rmax=700.0)
    with ht.Context(b, ht.Ranges(), threshold=2, max_hits=n) as ctx:
        ctx.fill(x, y, z)
        buf = torch.full((b.n_cells + 64,), -1, dtype=torch.int32, device="cuda")
        dst = buf[shift:shift + b.n_cells]
        torch.cuda.synchronize()
        ctx.matrix_into(dst)
        ctx.sync()
        got = buf.cpu().numpy()
        assert np.array_equal(got[shift:shift + b.n_cells].view(np.uint32), ctx.matrix().ravel())
        assert np.all(got[:shift] == -1) and np.all(got[shift + b.n_cells:] == -1)


@pytest.mark.parametrize("n_a", [64, 2048], ids=["ordinary", "compressible"])
def test_destroyed_beside_a_capture(ht, n_a):
    """A context is destroyed by one thread while another captures a stream: the
    capture stays valid, and the context's memory is given back."""
    import threading

    import torch
    b, r, T = ht.Binning(1, 2, n_a, 2048), ht.Ranges(), 3
    x, y, z = random_hits(600, n_a)
    dev = [torch.from_numpy(a).cuda() for a in (x, y, z)]
    M_ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
    pk_ref, n_ref = oracle.find_maxima(_ob(b), _orr(r), M_ref, T)
    out = torch.zeros(n_ref, 8, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = torch.cuda.Stream()
    with ht.Context(b, r, threshold=T, max_hits=600) as ctx:
        ctx.fill(*dev, stream=st)
        ctx.find_maxima(capacity=n_ref, out=out, count=cnt, stream=st)
        ctx.sync(stream=st)
        out.zero_()
        cnt.zero_()
        other = ht.Context(b, r, threshold=T, max_hits=600)
        other.fill(*dev)
        other.sync()
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st, capture_error_mode="thread_local"):
            ctx.fill(*dev, stream=st)
            t = threading.Thread(target=other.close)
            t.start()
            t.join()
            ctx.find_maxima(capacity=n_ref, out=out, count=cnt, stream=st)
        g.replay()
        torch.cuda.synchronize()
        assert int(cnt.item()) == n_ref
        assert_peaks_equal(out.cpu().numpy().view(ht.PEAK_DTYPE).reshape(-1), pk_ref)
        if n_a == 2048:
            assert torch.cuda.mem_get_info()[0] >= free + b.n_cells * 4
