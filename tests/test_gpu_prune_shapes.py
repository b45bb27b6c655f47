"""The cooperative prunes at the edges of their tiles, against the oracle bit for
bit: canonical prunes of any data, and prunes on the Gram tile of integer data
that bf16 holds exactly with fp32-exact dot products, where both decide every
test alike."""
import numpy as np
import pytest

from tests.pair import graphs_equal, make_pair

pytestmark = pytest.mark.gpu


def _rows(rng, n, m, integer):
    c = rng.normal(0, 8, size=(5, m))
    x = c[rng.integers(0, 5, n)] + rng.normal(size=(n, m))
    return (np.clip(np.rint(x), -60, 60) if integer else x).astype(np.float32)


def _rounds(g, o, rng, n, m, integer, R):
    for r in range(3):
        x = _rows(rng, 250 if r == 0 else 90, m, integer)
        g.insert(x)
        o.insert(x)
        dele = rng.choice(240, 60, replace=False).astype(np.uint32)
        assert g.delete(dele) == o.delete(dele)
        if r != 1:
            g.reclaim()
            o.reclaim()
        assert graphs_equal(g.export_graph(), o.dump(), R) == []


@pytest.mark.parametrize("m,metric,R,max_cand", [
    (1, "l2", 2, 0),
    (24, "l2", 9, 0),         # a second group of eight candidates with one member
    (100, "ip", 33, 128),     # the most rows of a cooperative canonical prune
    (127, "l2", 32, 64),
    (128, "l2", 64, 65),      # lists longer than a warp, folds of up to 127 candidates
    (129, "l2", 63, 129),     # prunes of more than 128 candidates keep the one-warp walk
    (260, "ip", 64, 0),
    (516, "l2", 8, 9),
])
def test_canonical_prunes_equal_oracle(oracle_mod, m, metric, R, max_cand):
    rng = np.random.default_rng(100 * m + R)
    g, o = make_pair(oracle_mod, m, metric, R, 800, build_beam=64, n_entry=32, max_cand=max_cand, max_batch=70)
    _rounds(g, o, rng, 800, m, False, R)


@pytest.mark.parametrize("m,metric,R,max_cand", [
    (64, "l2", 2, 33),
    (128, "ip", 32, 64),      # the largest one-warp tile
    (128, "l2", 33, 65),      # the smallest cooperative one
    (130, "l2", 32, 64),      # few rows, three column blocks
    (260, "ip", 64, 128),
    (768, "l2", 63, 0),
])
def test_tile_prunes_of_exact_data_equal_oracle(oracle_mod, m, metric, R, max_cand):
    rng = np.random.default_rng(100 * m + R)
    g, o = make_pair(oracle_mod, m, metric, R, 800, build_beam=64, n_entry=32, max_cand=max_cand, max_batch=70,
                     gram="tensor")
    _rounds(g, o, rng, 800, m, True, R)


@pytest.mark.parametrize("m,metric,R", [(24, "l2", 64), (130, "ip", 33)])
def test_canonical_offers_of_large_batches_equal_oracle(oracle_mod, m, metric, R):
    """More offers than the cooperative prunes take (64 per SM): a warp per list."""
    rng = np.random.default_rng(m)
    g, o = make_pair(oracle_mod, m, metric, R, 1600, build_beam=64, n_entry=32, max_batch=512)
    for n in (1100, 500):
        x = _rows(rng, n, m, False)
        g.insert(x)
        o.insert(x)
        assert graphs_equal(g.export_graph(), o.dump(), R) == []
