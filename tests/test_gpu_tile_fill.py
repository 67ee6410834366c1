"""The tile fill (one warp per tile, peaks found in the tile) against the
oracle at the edges of its shapes: passes of one row and of a remainder, a
single A bin, unit lists around the 128 lines a warp loads ahead, passes that
list up to 32, up to 127 and more cells, peaks on the rows where two passes
meet, the narrowest and the widest rows."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_parity import ht, _ob, _orr, assert_peaks_equal, random_hits  # noqa: F401

pytestmark = pytest.mark.gpu

# (n_theta, n_phi, n_a, n_b), hits, thresholds
SHAPES = [
    ((1, 1, 1, 64), 127, (1, 6)), ((1, 1, 2, 4), 128, (3, 30)), ((1, 2, 3, 32), 129, (2, 7)),
    ((1, 2, 5, 1024), 260, (1, 2)), ((2, 3, 13, 100), 900, (2, 4, 6)), ((1, 1, 9, 4096), 1500, (1, 2)),
    ((3, 2, 67, 256), 3000, (2, 3, 9)), ((1, 1, 33, 128), 2049, (10, 24)), ((4, 8, 130, 512), 33, (1, 2)),
    # rows that are not whole 16 bytes: passes start and end anywhere inside them
    ((1, 1, 1, 1), 50, (1, 20)), ((2, 1, 3, 2), 90, (2, 9)), ((1, 3, 7, 3), 200, (2, 12)), ((1, 2, 5, 1023), 260, (1, 2)),
    ((2, 3, 13, 101), 900, (2, 4, 6)), ((1, 1, 9, 4095), 1500, (1, 2)), ((3, 2, 67, 258), 3000, (2, 3, 9)),
]


@pytest.mark.parametrize("rows", [0, 1, 2, 8, 64], ids=lambda r: f"rows{r}")
@pytest.mark.parametrize("shape", SHAPES, ids=[str(s[0]) for s in SHAPES])
def test_tile_fill_shapes(ht, shape, rows):
    bins, n, thresholds = shape
    b, r = ht.Binning(*bins), ht.Ranges()
    x, y, z = random_hits(n, n, rmax=700.0)
    M_ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
    for T in thresholds:
        pk_ref, n_ref = oracle.find_maxima(_ob(b), _orr(r), M_ref, T)
        with ht.Context(b, r, threshold=T, max_hits=n) as ctx:
            ctx.set_tuning(fill_rows=rows)
            for _ in range(2):
                ctx.fill(x, y, z)
                pk, total = ctx.find_maxima(capacity=1 << 18)
                assert total == n_ref, T
                assert_peaks_equal(pk, pk_ref)
            assert np.array_equal(ctx.matrix(), M_ref)
            # the same passes without the writing: M_H stays what it was
            for _ in range(2):
                ctx.fill(x[:n // 2], y[:n // 2], z[:n // 2], peaks_only=True)
                ctx.fill(x, y, z, peaks_only=True)
                pk, total = ctx.find_maxima(capacity=1 << 18)
                assert total == n_ref, T
                assert_peaks_equal(pk, pk_ref)
            assert np.array_equal(ctx.matrix(), M_ref)


@pytest.mark.parametrize("n_b", [64, 61, 30])
def test_tile_fill_batch(ht, n_b):
    """Events of very different sizes (one empty) in one launch: the ranks run
    over all events' passes, and the counts are each event's own."""
    b, r, T = ht.Binning(2, 4, 37, n_b), ht.Ranges(), 3
    events = [random_hits(n, 50 + n) for n in (1, 0, 700, 31, 128, 2500, 5)]
    with ht.Batch(b, r, threshold=T, max_events=len(events), max_hits=4000, capacity=1 << 16) as B:
        for _ in range(3):   # captured after the first run
            pk, counts = B.run(*ht.Batch.concat(events))
            at = 0
            for e, (x, y, z) in enumerate(events):
                M_ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
                pk_ref, n_ref = oracle.find_maxima(_ob(b), _orr(r), M_ref, T)
                assert counts[e] == n_ref, e
                got = pk[at:at + n_ref]
                assert np.all(got["event"] == e)
                assert_peaks_equal(got, pk_ref)
                assert np.array_equal(B.matrix(e), M_ref)
                at += n_ref
            assert len(pk) == at


@pytest.mark.parametrize("S", [4, 16])
def test_sectors_count_edge_hits_once(ht, S):
    """Hits on the axes and diagonals, which are sector edges: the sectors'
    matrices are their phi bins of the unsplit one, the peaks the unsplit
    peaks."""
    from tests.test_gpu_parity import degenerate_hits
    x, y, z = degenerate_hits()
    b, r, T = ht.Binning(4, 16, 128, 100), ht.Ranges(), 3
    M_ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
    pk_ref, n_ref = oracle.find_maxima(_ob(b), _orr(r), M_ref, T)
    with ht.Sectors(b, r, threshold=T, n_sectors=S, max_hits=len(x)) as sec:
        sec.fill(x, y, z)
        pk, n = sec.find_maxima(capacity=1 << 18)
        assert n == n_ref
        assert_peaks_equal(pk, pk_ref)
        m = b.n_phi // S
        for k in range(S):
            assert np.array_equal(sec.matrix(k), M_ref[:, k * m:(k + 1) * m])


@pytest.mark.parametrize("rows", [0, 1, 2, 16], ids=lambda r: f"rows{r}")
@pytest.mark.parametrize("n_b", [96, 45])
def test_crowded_passes(ht, n_b, rows):
    """Many hits per slice (admission windows, crowded batches): the rows where
    two passes meet are compared after the fill.  Around the number of hits per
    slice that this begins at, with equal votes on both sides of an edge, and
    with counts above the capacity."""
    b, r = ht.Binning(2, 3, 53, n_b, 1, 1), ht.Ranges()
    # 9 admissions per hit, 6 slices, 192 hits per slice: from 128 hits on (n // 2 of them) for one event, from 384 for three
    for n in (254, 256, 383, 384, 3000):
        events = [random_hits(n // 2, n), random_hits(0, 1), random_hits(n - n // 2, n + 1)]
        for T in (1, 3, 9):
            ref = []
            for x, y, z in events:
                M_ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
                ref.append((M_ref, *oracle.find_maxima(_ob(b), _orr(r), M_ref, T)))
            with ht.Context(b, r, threshold=T, max_hits=n) as ctx:
                ctx.set_tuning(fill_rows=rows)
                for (x, y, z), (M_ref, pk_ref, n_ref) in zip(events, ref):
                    ctx.fill(x, y, z)
                    pk, total = ctx.find_maxima(capacity=1 << 16)
                    assert total == n_ref
                    assert_peaks_equal(pk, pk_ref)
                    assert np.array_equal(ctx.matrix(), M_ref)
                    ctx.fill(x, y, z)
                    pk, total = ctx.find_maxima(capacity=7)
                    assert total == n_ref
                    assert_peaks_equal(pk, pk_ref[:7])
            with ht.Batch(b, r, threshold=T, max_events=3, max_hits=n, capacity=1 << 16) as B:
                for _ in range(3):
                    pk, counts = B.run(*ht.Batch.concat(events))
                    assert list(counts[:3]) == [q[2] for q in ref]
                    at = 0
                    for e, (M_ref, pk_ref, n_ref) in enumerate(ref):
                        assert np.all(pk[at:at + n_ref]["event"] == e)
                        assert_peaks_equal(pk[at:at + n_ref], pk_ref)
                        at += n_ref


def test_edges_follow_the_runs_hits(ht):
    """A batch with room for many more hits than a run has: whether the rows
    where two passes meet are compared after the fill goes by the run's own hits
    (192 admissions per slice on average), directly and in the captured graphs,
    crowded and sparse runs in turn."""
    b, r, T = ht.Binning(2, 3, 53, 96), ht.Ranges(), 3
    runs = {}
    for n in (100, 2303, 2304, 9000):     # two events of 6 slices: from 2304 hits on
        evs = [random_hits(n // 3, n, rmax=700.0), random_hits(n - n // 3, n + 1, rmax=700.0)]
        ref = []
        for x, y, z in evs:
            M_ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
            ref.append((M_ref, *oracle.find_maxima(_ob(b), _orr(r), M_ref, T)))
        runs[n] = (evs, ref)
    with ht.Batch(b, r, threshold=T, max_events=2, max_hits=1 << 16, capacity=1 << 16) as B:
        for rep in range(3):
            for n in (100, 9000, 2303, 2304):
                evs, ref = runs[n]
                B.profile(rep == 0)
                pk, counts = B.run(*ht.Batch.concat(evs))
                if rep == 0:
                    assert B.profile_read()["k_edges"][0] == (n >= 2304), n
                assert list(counts) == [q[2] for q in ref]
                assert_peaks_equal(pk, np.concatenate([q[1] for q in ref]))
                for e in range(2):
                    assert np.array_equal(B.matrix(e), ref[e][0])


@pytest.mark.parametrize("peaks_only", [False, True])
def test_high_tiles_leave_the_sm_its_warps(ht, peaks_only):
    """Rows of 1024 bins: 16 to 64 rows per tile as asked for would leave an SM
    three warps, one or none; the fill takes lower ones and is as fast as 8 rows."""
    import torch
    from paper_1507_03074_gb300 import synth
    b, r = ht.Binning(*synth.PAPER_BINNING), ht.Ranges()
    ev = synth.paper_event(seed=11)
    d = [torch.from_numpy(a).cuda() for a in (ev.x, ev.y, ev.z)]
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with ht.Context(b, r, threshold=10, max_hits=ev.n_hits) as ctx:
        ctx.fill(*d)
        want, n_want = ctx.find_maxima(capacity=1 << 16)
        times = {}
        for rows in (8, 16, 32, 64):
            ctx.set_tuning(fill_rows=rows)
            assert ctx.get_tuning()["fill_rows"] == rows
            for n in (20, 100):       # warm, then timed
                t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                t0.record(st)
                for _ in range(n):
                    ctx.fill(*d, peaks_only=peaks_only, stream=st)
                t1.record(st)
                st.synchronize()
                times[rows] = t0.elapsed_time(t1) / n
            pk, n = ctx.find_maxima(capacity=1 << 16)
            assert n == n_want
            assert_peaks_equal(pk, want)
        assert max(times.values()) < 1.4 * times[8], times


def _one_slice(n, seed, phi=0.32):
    """n hits with one azimuth and one polar angle, as good as."""
    g = np.random.default_rng(seed)
    rad, ph, z = g.uniform(20, 1100, n), g.uniform(phi - 0.01, phi + 0.01, n), g.uniform(5, 12, n)
    return [a.astype(np.float32) for a in (rad * np.cos(ph), rad * np.sin(ph), z)]


# (n_theta, n_phi, n_a, n_b), uniform hits, hits in one slice, thresholds
CROWDED = [
    ((1, 1, 1, 64), 3000, 0, (2, 60)), ((1, 1, 2, 4096), 5000, 0, (1, 3)), ((1, 1, 3, 7), 2500, 0, (2, 500)),
    ((1, 2, 5, 1023), 4000, 0, (3, 9)), ((2, 2, 33, 200), 9000, 0, (4, 40)), ((1, 4, 129, 64), 8000, 0, (5, 80)),
    ((4, 10, 6, 333), 60000, 0, (6, 12)), ((3, 30, 41, 48), 100, 4000, (2, 30)), ((2, 3, 300, 1024), 900, 6000, (3, 5)),
    ((1, 1, 5, 64), 70000, 0, (40, 1500)), ((1, 64, 4, 96), 0, 513, (2, 9)), ((1, 64, 4, 96), 0, 512, (2, 9)),
]


@pytest.mark.parametrize("rows", [0, 1, 16], ids=lambda r: f"rows{r}")
@pytest.mark.parametrize("shape", CROWDED, ids=[str(s[:3]) for s in CROWDED])
def test_units_voted_by_whole_ctas(ht, shape, rows):
    """Units of so many hits that their passes are the whole CTA's: few rows and
    many hits, one crowded slice among sparse ones, more than 32 of them, on
    either side of the number of hits (512) that this begins at."""
    bins, n, one, thresholds = shape
    b, r = ht.Binning(*bins), ht.Ranges()
    parts = [random_hits(n, n + 1, rmax=900.0), _one_slice(one, one + 2)]
    x, y, z = (np.concatenate(v) for v in zip(*parts))
    M_ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
    for T in thresholds:
        pk_ref, n_ref = oracle.find_maxima(_ob(b), _orr(r), M_ref, T, cap=1 << 18)
        with ht.Context(b, r, threshold=T, max_hits=x.size) as ctx:
            ctx.set_tuning(fill_rows=rows)
            for po in (False, True, False, True):
                ctx.fill(x, y, z, peaks_only=po)
                pk, total = ctx.find_maxima(capacity=1 << 18)
                assert total == n_ref, (T, po)
                assert_peaks_equal(pk, pk_ref)
            assert np.array_equal(ctx.matrix(), M_ref)
            ctx.fill(x[:40], y[:40], z[:40])   # and a sparse fill after them
            M, _ = oracle.fill(_ob(b), _orr(r), x[:40], y[:40], z[:40])
            assert np.array_equal(ctx.matrix(), M)


def test_crowded_unit_in_a_batch(ht):
    """The crowded slice is the last event's, the first's, or each one's; sparse
    and crowded runs take turns on the captured graphs."""
    b, r, T = ht.Binning(2, 16, 30, 100), ht.Ranges(), 6
    sparse = [random_hits(40 + 30 * k, 300 + k, rmax=900.0) for k in range(5)]
    crowd = _one_slice(3000, 4)
    runs = [sparse, sparse[:4] + [crowd], [crowd] + sparse[:4], [crowd] * 5]
    refs = []
    for evs in runs:
        ref = []
        for x, y, z in evs:
            M_ref, _ = oracle.fill(_ob(b), _orr(r), x, y, z)
            ref.append((M_ref, *oracle.find_maxima(_ob(b), _orr(r), M_ref, T)))
        refs.append(ref)
    with ht.Batch(b, r, threshold=T, max_events=5, max_hits=1 << 15, capacity=1 << 17) as B:
        for rep in range(3):
            for po in (False, True):
                for evs, ref in zip(runs, refs):
                    pk, counts = B.run(*ht.Batch.concat(evs), peaks_only=po)
                    assert list(counts) == [q[2] for q in ref]
                    assert_peaks_equal(pk, np.concatenate([q[1] for q in ref]))
                    if not po:
                        for e in (0, 4):
                            assert np.array_equal(B.matrix(e), ref[e][0])
