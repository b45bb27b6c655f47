"""Ground truth on tensor cores (tcgen05 candidate pass + certified exact
rerank) against the CUDA-core exact kernel (bit-exact ids and distance
bits) and against the oracle's brute force, on the three mixture families:
integer data (exact in bf16: one bf16 segment), Gaussian data (hi/lo split)
and unit vectors under inner product.  Sizes span several 128-row tiles with
a ragged tail, a ragged query tile, and deleted rows."""
import dataclasses

import numpy as np
import pytest

from paper_2607_02543_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _pair_indices(w, n, deleted_every, **kw):
    from paper_2607_02543_gb300 import Index
    plan = W.make_plan(dataclasses.replace(W.scaled(w, n, n_queries=333), rounds=0))
    out = []
    for gt in ("default", "cuda_cores"):
        g = Index(w.dim, w.metric, w.degree, n + 10, build_beam=16, max_cand=32, gt=gt, **kw)
        g.insert(plan.base)
        if deleted_every:
            g.delete(np.arange(0, n, deleted_every, dtype=np.uint32))
        out.append(g)
    return plan, out


@pytest.mark.parametrize("wname,n,k,path", [
    ("int", 5_000 + 77, 10, "tensor"),
    ("gauss", 4_000 + 5, 10, "tensor_split"),
    ("unit", 3_000 + 31, 7, "tensor_split"),
    ("int", 300, 32, "tensor"),
    ("wide", 2_000 + 3, 10, "tensor_split"),    # 300-d: the query tile streams through the ring
    ("gist", 1_500 + 11, 10, "tensor_split"),   # 960-d non-negative mixture, streamed
])
def test_tensor_ground_truth_matches_exact(oracle_mod, wname, n, k, path):
    base = {"int": W.SIFT_LIKE_1M, "gauss": W.SMALL,
            "unit": dataclasses.replace(W.SMALL, metric="ip", kind="unit", dim=96),
            "wide": dataclasses.replace(W.SMALL, dim=300), "gist": W.GIST_LIKE_1M}[wname]
    plan, (gt_tc, gt_cc) = _pair_indices(base, n, 9)
    ti, td = gt_tc.ground_truth(plan.queries, k)
    info = gt_tc.ground_truth_info()
    ci, cd = gt_cc.ground_truth(plan.queries, k)
    assert gt_cc.ground_truth_info()["path"] == "cuda_cores"
    assert info["path"] == path
    np.testing.assert_array_equal(ti, ci)
    np.testing.assert_array_equal(td.view(np.uint32), cd.view(np.uint32))
    if k <= 16:   # with k = 32 = the candidate count there is no margin to certify
        assert info["fallback_queries"] <= len(plan.queries) // 10, info
    # the oracle ranks in fp64: equal ids up to fp32 ties, close distances
    o = oracle_mod.Oracle(base.dim, base.metric, base.degree, n + 10, build_beam=16)
    o.insert(plan.base)
    o.delete(np.arange(0, n, 9, dtype=np.uint32))
    oi, od = o.exact_knn(plan.queries, k)
    assert (ti == oi).mean() > 0.999
    assert np.allclose(td, od, rtol=1e-5, atol=1e-5)


def test_tensor_ground_truth_few_live_rows():
    """Fewer live rows than k: padded with NIL / +inf like the exact kernel."""
    from paper_2607_02543_gb300 import Index, NIL
    rng = np.random.default_rng(3)
    X = rng.integers(0, 255, size=(20, 128)).astype(np.float32)
    g = Index(128, "l2", 8, 100, build_beam=16)
    g.insert(X)
    g.delete(np.arange(0, 20, 2, dtype=np.uint32))
    ids, d = g.ground_truth(X[:50], 16)
    assert g.ground_truth_info()["path"] == "tensor"
    assert (ids[:, 10:] == NIL).all() and np.isinf(d[:, 10:]).all()
    assert set(ids[0, :10].tolist()) == set(range(1, 20, 2))


@pytest.mark.parametrize("n,nq,k,kind,dim", [
    (2_000 + 9, 1, 10, "gauss", 100),      # a block per query
    (2_000 + 9, 2_431, 10, "gauss", 128),
    (2_000 + 9, 2_500, 32, "gauss", 37),   # a warp per query; more candidate blocks than a lane keeps
    (9_000 + 1, 2_432, 1, "absgauss", 200),
    (33, 2_500, 5, "int", 128),
])
def test_rerank_team_shapes(n, nq, k, kind, dim):
    """A block or a warp per query, thresholds met by few or by many blocks: the exact kernel's bits."""
    from paper_2607_02543_gb300 import Index
    w = dataclasses.replace(W.scaled(W.SMALL, n, n_queries=nq), rounds=0, kind=kind, dim=dim, n_clusters=8)
    plan = W.make_plan(w)
    res = []
    for gt in ("default", "cuda_cores"):
        g = Index(dim, "l2", 16, n + 10, build_beam=16, max_cand=32, gt=gt)
        g.insert(plan.base)
        g.delete(np.arange(0, n, 7, dtype=np.uint32))
        res.append(g.ground_truth(plan.queries, k))
        if gt == "default":
            assert g.ground_truth_info()["fallback_queries"] == 0
    np.testing.assert_array_equal(res[0][0], res[1][0])
    np.testing.assert_array_equal(res[0][1].view(np.uint32), res[1][1].view(np.uint32))


@pytest.mark.parametrize("n,nq,k,metric,dim,integer", [
    (255, 1, 1, "l2", 32, True),           # one row tile, not full
    (257, 127, 32, "ip", 64, True),        # two row tiles, ties and zero keys of both signs
    (3_000, 129, 10, "l2", 129, False),    # two query tiles, rows longer than one column block
    (9_999, 609, 10, "l2", 100, True),     # the last row count at which the keys are written ...
    (20_481, 609, 10, "l2", 128, True),    # ... and the first beyond it
    (4_000, 1_217, 32, "ip", 300, False),  # the query tile streams; one warp per query
])
def test_rerank_by_row_keys(n, nq, k, metric, dim, integer):
    """Rows chosen by their own keys: the exact kernel's bits, with repeated and
    all-zero rows and whole blocks deleted."""
    from paper_2607_02543_gb300 import Index
    rng = np.random.default_rng(n + nq)
    c = rng.normal(0, 12, size=(7, dim))
    draw = lambda m: c[rng.integers(0, 7, m)] + rng.normal(0, 3, size=(m, dim))
    x, q = draw(n), draw(nq)
    if integer:
        x, q = np.clip(np.rint(x), -100, 100), np.clip(np.rint(q), -100, 100)
    x[rng.integers(0, n, n // 5)] = x[rng.integers(0, n, n // 5)]
    x[::17] = 0.0
    q[::5] = 0.0
    x, q = x.astype(np.float32), q.astype(np.float32)
    dele = np.concatenate([np.arange(32, 96), np.arange(97, n, 11)]).astype(np.uint32)
    res = []
    for gt in ("default", "cuda_cores"):
        g = Index(dim, metric, 8, n + 10, build_beam=16, max_cand=16, gt=gt)
        g.insert(x)
        g.delete(dele)
        res.append(g.ground_truth(q, k))
    np.testing.assert_array_equal(res[0][0], res[1][0])
    np.testing.assert_array_equal(res[0][1].view(np.uint32), res[1][1].view(np.uint32))


def test_close_gives_the_workspaces_back():
    """Ground truth, seeding and round workspaces (about 60 MB here) do not outlive their index."""
    import torch
    from paper_2607_02543_gb300 import Index
    x = np.random.default_rng(1).normal(size=(4_000, 128)).astype(np.float32)
    free = []
    for _ in range(3):
        g = Index(128, "l2", 32, 5_000, build_beam=32, n_entry=512, mode="lockfree")
        g.insert(x)
        g.ground_truth(x, 10)
        g.search(x, 10, 32)
        g.close()
        free.append(torch.cuda.mem_get_info()[0])
    assert free[0] - free[2] < 16 << 20, free   # the first pass pays for the context's own allocations
