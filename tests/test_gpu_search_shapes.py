"""The BeamSearch kernels at the edges of their row lengths, degrees, beams and
batch sizes, against the oracle (fp32) and against the fp32 search (BF16 keys of
integer data, which are exact)."""
import numpy as np
import pytest

from tests.pair import make_pair

pytestmark = pytest.mark.gpu


def _data(rng, n, m, integer):
    c = rng.normal(0, 10, size=(6, m))
    x = c[rng.integers(0, 6, n)] + rng.normal(size=(n, m))
    return (np.rint(x) if integer else x).astype(np.float32)


@pytest.mark.parametrize("m,metric,R,beam,k", [
    (1, "l2", 8, 1, 1),          # one element, one beam entry
    (3, "ip", 5, 31, 7),
    (127, "l2", 32, 32, 32),     # the last row of the 8-lane form, beam of one chunk
    (128, "ip", 33, 33, 10),     # two halves of a slab
    (129, "l2", 32, 64, 10),     # the first row of the whole-warp form
    (260, "ip", 64, 96, 20),     # three column blocks, the last one lane wide
    (513, "l2", 16, 256, 256),   # the largest beam, k = beam
    (1030, "l2", 33, 40, 5),
])
def test_search_equals_oracle(oracle_mod, m, metric, R, beam, k):
    rng = np.random.default_rng(1000 * m + R)
    n = 400
    x, q = _data(rng, n, m, False), _data(rng, 67, m, False)
    g, o = make_pair(oracle_mod, m, metric, R, n, build_beam=24, n_entry=16)
    g.insert(x)
    o.insert(x)
    dele = np.arange(0, n, 9, dtype=np.uint32)
    assert g.delete(dele) == o.delete(dele)   # tombstones relay in the searches
    for nq in (1, 67):
        gi, gd = g.search(q[:nq], k, beam)
        oi, od = o.search(q[:nq], k, beam)
        np.testing.assert_array_equal(gi, oi)
        np.testing.assert_array_equal(gd.view(np.uint32), od.view(np.uint32))


@pytest.mark.parametrize("m,nq", [(127, 40), (128, 2600), (129, 40), (320, 2600)])
def test_reduced_rows_of_integer_data_equal_fp32(m, nq):
    from paper_2607_02543_gb300 import Index
    rng = np.random.default_rng(m)
    n = 1500
    x, q = _data(rng, n, m, True), _data(rng, nq, m, True)
    g = Index(m, "l2", 32, n, build_beam=32, n_entry=64, copies=("bf16",))
    g.insert(x)
    ref = g.search(q, 10, 48)
    g.set_search_precision("bf16")
    for tensor in (True, False):
        g.set_search_keys(tensor)
        for shape in (None, (2, 6, 2), (32, 12, 8)):
            if shape:
                g.set_search_tuning(*shape)
            ids, d = g.search(q, 10, 48)
            np.testing.assert_array_equal(ids, ref[0])
            np.testing.assert_array_equal(d.view(np.uint32), ref[1].view(np.uint32))
