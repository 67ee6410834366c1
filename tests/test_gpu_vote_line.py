"""The votes' linear model (the bin of a vote without a division, with the
rule of the ABI next to a bin edge) against the oracle, where the two could
part: votes exactly on bin edges, steep lines (y near 0), ranges far from the
origin (the model's error exceeds half a bin and the rule decides every
vote), the smallest and the widest row that the tile fills hold."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_parity import ht, _ob, _orr, assert_peaks_equal, random_hits, run_gpu  # noqa: F401

pytestmark = pytest.mark.gpu


def on_edges(n, seed):
    """Hits whose votes fall on bin edges of power-of-two bins: y a power of
    two and whole x, so that every B is exact."""
    rng = np.random.default_rng(seed)
    y = np.float32(2.0) ** rng.integers(3, 8, n).astype(np.float32) * rng.choice(np.float32([-1, 1]), n)
    return (rng.integers(-64, 65, n).astype(np.float32), y.astype(np.float32),
            rng.uniform(-300, 300, n).astype(np.float32))


def steep(n, seed):
    """Hits with |y| from 1e-6 of |x| up."""
    x, y, z = random_hits(n, seed)
    f = np.exp(np.random.default_rng(seed).uniform(np.log(1e-6), 0, n)).astype(np.float32)
    return x, (y * f).astype(np.float32), z


def distant(n, seed):
    """Hits at y around 4e6, whose B is around 2e6."""
    rng = np.random.default_rng(seed)
    return tuple(rng.uniform(a, b, n).astype(np.float32) for a, b in ((-1e3, 1e3), (4.0e6, 4.0002e6), (-1e6, 1e6)))


CASES = [
    ("edges", (2, 4, 64, 64), dict(a_min=-128.0, a_max=128.0, b_min=-256.0, b_max=256.0), 3, on_edges(900, 1)),
    ("edges_odd_rows", (1, 4, 33, 128), dict(a_min=-64.5, a_max=67.5, b_min=-64.0, b_max=64.0), 3, on_edges(900, 2)),
    ("steep", (2, 4, 128, 256), {}, 3, steep(3000, 3)),
    ("far_ranges", (1, 2, 40, 300), dict(a_min=1.0e5, a_max=1.00004e5, b_min=-3.0e6, b_max=3.0e6), 2,
     random_hits(800, 4)),
    ("fine_far_ranges", (1, 2, 24, 512), dict(a_min=-100.0, a_max=100.0, b_min=2.0e6, b_max=2.0001e6), 2,
     distant(1500, 5)),
    ("one_bin", (1, 2, 5, 1), {}, 2, random_hits(300, 6)),
    ("widest_row", (1, 2, 9, 4096), {}, 2, random_hits(2500, 7)),
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_vote_line_matches_the_rule(ht, case):
    name, bins, rng, T, (x, y, z) = case
    b, r = ht.Binning(*bins), ht.Ranges(**rng)
    M_ref, votes = oracle.fill(_ob(b), _orr(r), x, y, z)
    pk_ref, n_ref = oracle.find_maxima(_ob(b), _orr(r), M_ref, T)
    assert votes > 0
    for tuning in (None, dict(fill_fused_scan=2), dict(bin_cluster=2)):
        M, pk, n, _ = run_gpu(ht, b, r, T, x, y, z, tuning=tuning)
        assert np.array_equal(M, M_ref), tuning
        assert n == n_ref
        assert_peaks_equal(pk, pk_ref)
