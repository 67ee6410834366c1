"""Accumulating fills on both sides of the line between reductions into M_H
and the fill that reads and writes all of it, against the oracle: odd rows,
admission windows, ranges that cut hits off, fills of no hits, the first fill
being an accumulating one."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_parity import ht, _ob, _orr, assert_peaks_equal, random_hits  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [((2, 4, 64, 64), {}), ((3, 5, 37, 29), {}), ((4, 16, 128, 131, 1, 1), {}), ((1, 1, 33, 257), {}),
         ((3, 6, 80, 64, 1, 2), dict(theta_min=0.4, theta_max=2.6, phi_min=-2.0, phi_max=1.5))]


@pytest.mark.parametrize("case", CASES, ids=[str(c[0]) for c in CASES])
def test_accumulating_fills(ht, case):
    bins, rng = case
    b, r, T = ht.Binning(*bins), ht.Ranges(**rng), 3
    line = b.n_cells // 6 // b.n_a   # hits at which the votes of one slice each reach the line
    cuts = np.cumsum([0, 1, max(line // 9, 1), 0, 40, max(line // 9, 1) + 1, line + 1, 31, 2 * line + 5])
    x, y, z = random_hits(int(cuts[-1]), 91)
    M = np.zeros(b.shape(), np.uint32)
    with ht.Context(b, r, threshold=T, max_hits=int(cuts[-1])) as ctx:
        for k, (i, j) in enumerate(zip(cuts, cuts[1:])):
            ctx.fill(x[i:j], y[i:j], z[i:j], accumulate=True)
            M += oracle.fill(_ob(b), _orr(r), x[i:j], y[i:j], z[i:j])[0]
            assert np.array_equal(ctx.matrix(), M), k
            pk_ref, n_ref = oracle.find_maxima(_ob(b), _orr(r), M, T)
            pk, n = ctx.find_maxima(capacity=1 << 18)
            assert n == n_ref, k
            assert_peaks_equal(pk, pk_ref)
