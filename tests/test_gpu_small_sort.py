"""Rounds whose sorts lie at either side of the one-block form (4096 keys):
deletes of unordered ids with repeats, and deterministic offers and repair
pairs of as many slots, against the oracle bit for bit."""
import numpy as np
import pytest

from tests.pair import graphs_equal, make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 2, 128, 129])      # 129 x 32 slots: more than one block takes
@pytest.mark.parametrize("n_ids", [1, 33, 4096, 4097])
def test_sorted_rounds_equal_oracle(oracle_mod, batch, n_ids):
    rng = np.random.default_rng(n_ids + batch)
    n, m, R = 1200, 8, 32
    g, o = make_pair(oracle_mod, m, "l2", R, 1400, build_beam=32, n_entry=16, max_batch=600)
    x = rng.normal(size=(n + batch, m)).astype(np.float32)
    g.insert(x[:n])
    o.insert(x[:n])
    dele = rng.choice(128, n_ids).astype(np.uint32) * 7   # at most 128 distinct, repeats, no order
    assert g.delete(dele) == o.delete(dele)
    assert graphs_equal(g.export_graph(), o.dump(), R) == []
    g.insert(x[n:])
    o.insert(x[n:])
    assert graphs_equal(g.export_graph(), o.dump(), R) == []
