"""Matrices of more than 2 GiB: the fills and scans whose CTAs own ranges work
through them in windows.  Every such fill and scan against the tile fill (which
the other tests compare with the oracle), sampled slices at the windows' ends
against the oracle, and the time of a scan over many windows."""
import numpy as np
import pytest

import oracle
from paper_1507_03074_gb300 import synth
from tests.test_gpu_parity import ht, _ob, _orr, assert_peaks_equal, random_hits  # noqa: F401

pytestmark = pytest.mark.gpu

TUNINGS = [dict(fill_fused_scan=1), dict(fill_fused_scan=2), dict(fill_fused_scan=2, scan_kind=1),
           dict(fill_fused_scan=3), dict(fill_fused_scan=4), dict(fill_fused_scan=1, fill_rows=8, fill_threads=256)]


def _device(ev):
    import torch
    return [torch.from_numpy(a).cuda() for a in ev]


@pytest.mark.parametrize("n_b", [2048, 2047])
def test_windows_of_one_event(ht, n_b):
    import torch
    b, r, T = ht.Binning(5, 64, 1024, n_b), ht.Ranges(), 2   # 2.5 GiB: 256 slices (one more for 2047) and the rest
    ev = random_hits(20000, 7, rmax=900.0)
    win = (2 << 30) // (b.n_a * b.n_b * 4)
    d = _device(ev)
    ref, M = (torch.zeros(b.n_cells, dtype=torch.int32, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    with ht.Context(b, r, threshold=T, max_hits=40000) as ctx:
        ctx.fill(*d)
        pk_ref, n_ref = ctx.find_maxima(capacity=1 << 20)
        assert n_ref > 10000
        ctx.matrix_into(ref)
        ctx.sync()
        some = [0, win - 1, win, b.n_theta * b.n_phi - 1]
        got = ref.view(b.n_theta * b.n_phi, b.n_a, b.n_b)[some].cpu().numpy().view(np.uint32)
        want = oracle.fill_slices(_ob(b), _orr(r), *ev, some)
        want = want[0] if isinstance(want, tuple) else want
        assert np.array_equal(got, np.asarray(want).reshape(got.shape))
        # the scan alone
        pk, n = ctx.find_maxima(capacity=1 << 20)
        assert n == n_ref
        assert_peaks_equal(pk, pk_ref)
        for tuning in TUNINGS if n_b == 2048 else TUNINGS[:2]:
            ctx.set_tuning(**tuning)
            ctx.set_matrix(torch.full((b.n_cells,), 7, dtype=torch.int32, device="cuda"))
            torch.cuda.synchronize()
            ctx.fill(*d)
            for _ in range(2):   # the fill's own peaks (where it lists them), and the scan's
                pk, n = ctx.find_maxima(capacity=1 << 20)
                assert n == n_ref, tuning
                assert_peaks_equal(pk, pk_ref)
            ctx.matrix_into(M)
            ctx.sync()
            assert torch.equal(M, ref), tuning
        # accumulation by the private tiles (all at once: more votes than a sixth of the cells, else one by one)
        ctx.set_tuning()
        ctx.fill(*[t[:1] for t in d])
        ctx.fill(*[t[1:] for t in d], accumulate=True)
        ctx.matrix_into(M)
        pk, n = ctx.find_maxima(capacity=1 << 20)
        assert n == n_ref and torch.equal(M, ref)
        assert_peaks_equal(pk, pk_ref)


def test_windows_accumulate_by_tiles(ht):
    """So many votes that an accumulating fill goes through the private tiles."""
    import torch
    b, r = ht.Binning(3, 16, 2732, 4096), ht.Ranges()   # 2 GiB and a little
    assert b.n_cells * 4 > 2 << 30
    ev = random_hits(70000, 9, rmax=900.0)
    d = _device(ev)
    ref, M = (torch.zeros(b.n_cells, dtype=torch.int32, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    with ht.Context(b, r, threshold=30, max_hits=70000) as ctx:
        ctx.fill(*d)
        ctx.matrix_into(ref)
        ctx.fill(*[t[:500] for t in d])
        ctx.profile(True)
        before = ctx.launches
        ctx.fill(*[t[500:] for t in d], accumulate=True)
        assert ctx.profile_read()["k_fill_priv"][0] == 2 and ctx.launches - before == 4
        ctx.matrix_into(M)
        ctx.sync()
        assert torch.equal(M, ref)


@pytest.mark.parametrize("n_events", [8, 9, 17, 1])
def test_windows_of_a_batch(ht, n_events):
    b, r, T = ht.Binning(*synth.PAPER_BINNING), ht.Ranges(), 4   # eight events to a window
    evs = [random_hits(700 - 150 * (k % 5), 200 + k, rmax=900.0) for k in range(n_events)]
    x, y, z, off = ht.Batch.concat(evs)
    with ht.Batch(b, r, threshold=T, max_events=17, max_hits=20000, capacity=1 << 18) as B:
        pk_ref, c_ref = B.run(x, y, z, off)
        assert c_ref.sum() > 0
        M_ref = B.matrix(n_events - 1)
        pk1, n1 = None, 0
        with ht.Context(b, r, threshold=T, max_hits=20000) as ctx:
            ctx.fill(*evs[-1])
            pk1, n1 = ctx.find_maxima(capacity=1 << 18)
        assert n1 == c_ref[-1]
        assert_peaks_equal(pk_ref[len(pk_ref) - n1:], pk1)
        for tuning in TUNINGS:
            B.set_tuning(**tuning)
            for _ in range(2):   # direct, then the captured graph
                pk, counts = B.run(x, y, z, off)
                assert np.array_equal(counts, c_ref), tuning
                assert np.array_equal(pk, pk_ref), tuning
            assert np.array_equal(B.matrix(n_events - 1), M_ref)
        B.set_tuning()
        pk, counts = B.run(x, y, z, off, naive=True)
        assert np.array_equal(counts, c_ref) and np.array_equal(pk, pk_ref)


def test_scan_of_many_windows_is_streamed(ht):
    """15 GiB: the scan reads them at 5 TB/s or more (in ordinary memory 6.5; with
    the CTAs' ranges spread over the whole, 3.3)."""
    import torch
    b, r = ht.Binning(15, 64, 2048, 2048), ht.Ranges()
    ev = synth.make_event(*synth.split_hits(20000), seed=2)
    out = torch.zeros(1 << 16, 8, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = torch.cuda.Stream()
    with ht.Context(b, r, threshold=10, max_hits=20000) as ctx:
        ctx.fill(ev.x, ev.y, ev.z, stream=st)
        ctx.find_maxima(capacity=1 << 16, out=out, count=cnt, stream=st)
        st.synchronize()
        n_ref, ref = int(cnt.item()), out.clone()
        times = []
        for _ in range(5):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record(st)
            ctx.find_maxima(capacity=1 << 16, out=out, count=cnt, stream=st)
            t1.record(st)
            st.synchronize()
            times.append(t0.elapsed_time(t1))
            assert int(cnt.item()) == n_ref and torch.equal(out[:n_ref], ref[:n_ref])
        assert b.n_cells * 4 / min(times) / 1e9 > 5.0, times
