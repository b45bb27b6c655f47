"""Measured cases of the index: what a program that keeps a dynamic nearest-neighbour index has it do.

Four kinds of pass, each through the public `Index` class:
  query  one batch of k-NN queries on a built index (etale_search, or a captured query graph);
  truth  the exact k nearest live nodes of a query batch (etale_ground_truth);
  round  one churn round: delete, insert, reclaim, then a query batch on the updated graph (eager
         calls, or the recorded round graph);
  load   an index built from empty by one bulk insert, then queried.

The data are the Gaussian mixtures of `workloads.py` (integer-valued, Gaussian, unit-length and
non-negative), drawn on the GPU, with its dimensions, degrees, beams and cluster spacing; the index
options are the library's defaults except where the benchmark's configurations set them (build beam,
max_cand, entry-set size, lock-free mode, precisions).
"""
import math

import numpy as np
import torch

from paper_2607_02543_gb300 import Index

DEV = "cuda"


def _rounds(case):
    """Id budget of a `round` case, in rounds: ids are never reused, so a program sizes the budget for
    the life of the index and moves to a fresh one when it is spent."""
    if case["what"] != "round":
        return 0
    return min(1200, max(100, 160_000_000 // (case["churn"] * case["dim"])))


def _window(case):
    """Rows are drawn for this many rounds and cycled: long enough that a row comes back only after its
    first copy was deleted."""
    return min(_rounds(case), 2 + case["n"] // case["churn"]) if case["what"] == "round" else 0


def _case(name, what, kind, n, dim, **over):
    c = dict(name=name, what=what, kind=kind, n=n, dim=dim, clusters=256, metric="l2", degree=32, mode="lockfree",
             build_beam=64, max_cand=64, n_entry=1024, nq=1000, k=10, beam=64, prec="fp32", path="call", host=False,
             churn=0)
    c.update(over)
    return c


def listed():
    return [
        # one interactive query from host memory on a small default index: pure latency
        _case("query-1-int128-100k", "query", "int", 100_000, 128, clusters=64, nq=1, host=True),
        # the query batch of a service beside its updates (the concurrent-latency measurement's batch size)
        _case("query-1000-int128-1m", "query", "int", 1_000_000, 128, build_beam=128, n_entry=4096, beam=128),
        # the benchmark's throughput batch: 10,000 queries on the SIFT-shaped index at its beam
        _case("query-10k-int128-1m", "query", "int", 1_000_000, 128, build_beam=128, n_entry=4096, nq=10_000, beam=144),
        # text-embedding search: inner product, wide rows, degree 64, BF16 rows with an exact rerank
        _case("query-4k-ip768-bf16", "query", "unit", 50_000, 768, clusters=64, metric="ip", degree=64, max_cand=128,
              nq=4096, prec="bf16"),
        # GIST-shaped rows through one captured query graph whose batch size changes from call to call
        _case("query-1537-d960-graph", "query", "absgauss", 50_000, 960, clusters=64, nq=1537, k=32, beam=96,
              path="graph"),
        # a row length that is no multiple of the tile sizes, FP8 rows, more neighbours per query
        _case("query-4099-d100-fp8", "query", "gauss", 100_000, 100, clusters=64, nq=4099, k=20, beam=128, prec="fp8"),
        # recall measurement of the SIFT-shaped index (integer data: exact in bf16)
        _case("truth-10k-int128-300k", "truth", "int", 300_000, 128, nq=10_000),
        # recall measurement on wide real-valued rows (GIST-shaped), an uneven batch
        _case("truth-2003-d960-40k", "truth", "absgauss", 40_000, 960, clusters=64, nq=2003),
        # the benchmark's churn round (1% deleted, 1% inserted, reclaim, 10,000 queries) as one recorded graph
        _case("round-recorded-int128-1m", "round", "int", 1_000_000, 128, build_beam=128, n_entry=4096, nq=10_000,
              beam=144, churn=10_000, path="graph"),
        # embedding churn through the eager calls, with the BF16 form of inserts and queries
        _case("round-500-ip768-50k", "round", "unit", 50_000, 768, clusters=64, metric="ip", degree=64, max_cand=128, nq=1000,
              prec="bf16", churn=500),
        # small deterministic rounds fed from host memory (the parity workload's sizes)
        _case("round-100-gauss128-det", "round", "gauss", 10_000, 128, clusters=64, mode="deterministic", max_cand=128,
              churn=100, host=True),
        # the first load of the SIFT-shaped index: one bulk insert from empty
        _case("load-300k-int128", "load", "int", 300_000, 128, build_beam=128, n_entry=4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same four kinds over their whole ranges of size, shape, precision and path."""
    what = rng.choice(["query", "query", "query", "truth", "round", "round", "load"])
    kind, dims, metric, degree = rng.choice([("int", (64, 128), "l2", 32), ("int", (128, 160), "l2", 32),
                                             ("gauss", (37, 128), "l2", 32), ("gauss", (96, 100), "l2", 24),
                                             ("unit", (256, 768), "ip", 64), ("absgauss", (320, 960), "l2", 32)])
    if what == "load":   # many sub-batches of a hundredth of the capacity each: rows of ordinary width
        kind, dims, metric, degree = rng.choice([("int", (64, 160), "l2", 32), ("gauss", (37, 128), "l2", 32)])
    dim = rng.choice([dims[0], dims[1], rng.randint(dims[0], dims[1])])
    n = _log(rng, 10_000, min(600_000, 50_000 if degree == 64 else 150_000 if what == "load" else 64_000_000 // dim))
    entries = rng.choice([1024, 1024, 4096])
    c = dict(what=what, kind=kind, n=n, dim=dim, clusters=max(16, min(n // 1000, entries // 16)), metric=metric,
             degree=degree, mode="lockfree" if degree == 64 else rng.choice(["lockfree", "deterministic"]),
             build_beam=rng.choice([64, 64, 128]), max_cand=128 if degree == 64 else 64, n_entry=entries,
             k=rng.choice([1, 5, 10, 20]), beam=rng.choice([48, 64, 96, 128, 144]), prec="fp32", path="call",
             host=rng.random() < 0.25, churn=0)
    if what == "truth":
        c["nq"] = min(_log(rng, 1, 10_000), max(1, 90_000_000_000 // (n * dim)))
    elif what == "query":
        c["nq"] = min(_log(rng, 1, 16_384), 16_384 * 128 // max(128, dim))
        c["prec"] = rng.choice(["fp32", "fp32", "bf16", "fp8"])
        c["path"] = rng.choice(["call", "call", "graph"])
    else:
        c["nq"] = _log(rng, 100, 1000)
        if what == "round":
            c["churn"] = _log(rng, max(16, n // 1000), n // 100)
            c["prec"] = "bf16" if degree == 64 else "fp32"
    if c["path"] == "graph":
        c["host"] = False
    return c


# ---- data -------------------------------------------------------------------
def _mixture(case, g):
    """(the mixture's centres, a function drawing n of its points), as in workloads.Mixture."""
    m, kind, k = case["dim"], case["kind"], case["clusters"]
    if kind == "int":
        cen = 255.0 * torch.rand(k, m, generator=g, device=DEV)
    else:
        cen = torch.randn(k, m, generator=g, device=DEV)
        cen = cen / cen.norm(dim=1, keepdim=True) if kind == "unit" else 10.0 * cen
        cen = cen.abs() if kind == "absgauss" else cen

    def points(n):
        out = torch.empty(n, m, device=DEV)
        for lo in range(0, n, 1 << 18):
            b = min(n - lo, 1 << 18)
            c = cen[torch.randint(0, k, (b,), generator=g, device=DEV)]
            z = torch.randn(b, m, generator=g, device=DEV)
            if kind == "int":
                p = (c + 20.0 * z).round_().clamp_(0.0, 255.0)
            elif kind == "unit":
                p = c + (0.3 / math.sqrt(m)) * z
                p = p / p.norm(dim=1, keepdim=True)
            else:
                p = (c + z).abs_() if kind == "absgauss" else c + z
            out[lo:lo + b] = p
        return out

    return points


def _inputs(case, seed):
    """The base rows, the queries, the order in which base ids are deleted and the rows to insert."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    points = _mixture(case, g)
    x, q = points(case["n"]), points(case["nq"])
    if case["what"] != "round":
        return x, q, None, None
    order = torch.randperm(case["n"], generator=g, device=DEV).to(torch.int32)
    return x, q, order, points(_window(case) * case["churn"])


def _index(case):
    n = case["n"] + _rounds(case) * case["churn"]
    copies = () if case["prec"] == "fp32" else (case["prec"],)
    return Index(case["dim"], case["metric"], case["degree"], n, build_beam=case["build_beam"],
                 max_cand=case["max_cand"], n_entry=case["n_entry"], mode=case["mode"], copies=copies)


def prepare(case, seed):
    x, q, order, fresh = _inputs(case, seed)
    st = dict(case=case, seed=seed, q=q.cpu().numpy() if case["host"] else q)
    if case["what"] == "load":
        st["x"] = x.cpu().numpy() if case["host"] else x
        return st
    ix = _index(case)
    ix.insert(x)
    ix.set_search_precision(case["prec"])
    st["ix"] = ix
    if case["what"] == "query" and case["path"] == "graph":
        # the buffers hold the largest batch of the service; this call's batch size is on the device
        cap = 1 << max(5, (case["nq"] - 1).bit_length())
        buf = torch.zeros(cap, case["dim"], device=DEV)
        buf[:case["nq"]] = q
        ids = torch.zeros(cap, case["k"], dtype=torch.int32, device=DEV)
        dist = torch.zeros(cap, case["k"], device=DEV)
        size = torch.tensor([case["nq"]], dtype=torch.int32, device=DEV)
        torch.cuda.synchronize()
        st.update(buf=buf, out=(ids, dist), size=size, graph=ix.search_graph(buf, ids, dist, size, case["k"], case["beam"]))
    if case["what"] == "round":
        ix.set_insert_precision(case["prec"] if case["prec"] == "bf16" else "fp32")
        # victims: the base ids in random order, then the inserted ids, oldest first
        later = torch.arange(case["n"], case["n"] + _rounds(case) * case["churn"], dtype=torch.int32, device=DEV)
        victims = torch.cat([order, later])
        st.update(step=0, victims=victims, fresh=fresh)
        if case["host"]:
            st.update(victims=victims.cpu().numpy().view(np.uint32), fresh=fresh.cpu().numpy())
        if case["path"] == "graph":
            b = case["churn"]
            dele, ins = victims[:b].clone(), fresh[:b].clone()
            ids = torch.zeros(case["nq"], case["k"], dtype=torch.int32, device=DEV)
            dist = torch.zeros(case["nq"], case["k"], device=DEV)
            torch.cuda.synchronize()
            st.update(dele=dele, ins=ins, out=(ids, dist),
                      graph=ix.round_graph(dele, ins, st["q"], (ids, dist), k=case["k"], beam=case["beam"]))
    return st


def run(st):
    c = st["case"]
    k, beam = c["k"], c["beam"]
    if c["what"] == "load":
        ix = _index(c)
        new = ix.insert(st["x"])
        ids, dist = ix.search(st["q"], k, beam)
        ix.close()
        return {"new": new, "ids": ids, "dists": dist}
    ix = st["ix"]
    if c["what"] == "truth":
        ids, dist = ix.ground_truth(st["q"], k)
        return {"ids": ids, "dists": dist}
    if c["what"] == "query":
        if c["path"] == "graph":
            st["graph"].launch()
            return {"ids": st["out"][0][:c["nq"]], "dists": st["out"][1][:c["nq"]]}
        ids, dist = ix.search(st["q"], k, beam)
        return {"ids": ids, "dists": dist}
    if st["step"] == _rounds(c):
        # the id budget is spent: a fresh index from the start of the stream
        for h in ("graph", "ix"):
            if h in st:
                st.pop(h).close()
        st.update(prepare(c, st["seed"]))
        ix = st["ix"]
    b, i = c["churn"], st["step"]
    j = i % _window(c)
    dele, ins = st["victims"][i * b:(i + 1) * b], st["fresh"][j * b:(j + 1) * b]
    st["step"] = i + 1
    if c["path"] == "graph":
        st["dele"].copy_(dele)
        st["ins"].copy_(ins)
        st["graph"].launch()
        return {"ids": st["out"][0], "dists": st["out"][1]}
    gone = ix.delete(dele)
    new = ix.insert(ins)
    ix.reclaim()
    ids, dist = ix.search(st["q"], k, beam)
    return {"deleted": gone, "new": new, "ids": ids, "dists": dist}


# ---- what a pass cannot do without --------------------------------------------
def work(case):
    n, m, R, nq, k = case["n"], case["dim"], case["degree"], case["nq"], case["k"]
    if case["what"] == "truth":
        return {"bytes": 4.0 * m * (n + nq) + 8.0 * nq * k, "flops": 2.0 * n * nq * m}

    def walks(count, beam, row):
        # each walk expands about `beam` lists and scores about three in eight of their entries as new;
        # however many walks there are, no list and no row has to be read twice
        lists, rows = min(count * beam, n), min(count * beam * 0.375 * R, n)
        return lists * (8.0 + 8.0 * R) + rows * (row + 8.0), 3.0 * m * (count * beam * 0.375 * R + count * case["n_entry"])

    row = {"fp32": 4.0 * m, "bf16": 2.0 * m, "fp8": 1.0 * m}[case["prec"]]
    by, fl = walks(nq, case["beam"], row)
    by += 4.0 * m * (nq + min(n, case["n_entry"])) + 8.0 * nq * k
    if case["what"] == "query":
        return {"bytes": by, "flops": fl}
    b = n if case["what"] == "load" else case["churn"]
    ib, ifl = walks(b, case["build_beam"], row)
    # inserts: the rows in and stored, the new lists, and the lists that gain an edge
    by += ib + 8.0 * m * b + 8.0 * R * b + 16.0 * R * min(b * R, n)
    fl += ifl + 3.0 * m * b * case["max_cand"] * 4
    if case["what"] == "round":
        # deletes: the rows around each deleted node and its neighbours' lists; reclaim: every list once
        by += 4.0 * m * min(b * R, n) + 16.0 * R * min(b * R, n) + (8.0 + 8.0 * R) * n
        fl += 3.0 * m * b * R * R / 2
    return {"bytes": by, "flops": fl}


# ---- the answer in 64 bits ------------------------------------------------------
def exact(case, seed):
    """The true k nearest distances among the live rows, in 64 bits (ids and counts have no such value)."""
    x, q, order, fresh = _inputs(case, seed)
    if case["what"] == "round":
        b = case["churn"]
        x = torch.cat([x[order[b:].long()], fresh[:b]])
    k, keep, ip = case["k"], case["k"] + 48, case["metric"] == "ip"
    norm = torch.zeros(x.shape[0], device=DEV) if ip else (x * x).sum(1)
    best = torch.empty(q.shape[0], k, dtype=torch.float64, device=DEV)
    per = max(1, min(512, (1 << 28) // x.shape[0]))
    for lo in range(0, q.shape[0], per):
        qq = q[lo:lo + per]
        key = torch.addmm(norm, qq, x.t(), alpha=-1.0 if ip else -2.0)
        near = x[key.topk(keep, dim=1, largest=False).indices].double()
        d = 1.0 - torch.einsum("qm,qkm->qk", qq.double(), near) if ip else (near - qq.double()[:, None]).square().sum(2)
        best[lo:lo + per] = d.topk(k, dim=1, largest=False).values
    full = {"ids": None, "dists": best}
    if case["what"] == "load" or (case["what"] == "round" and case["path"] == "call"):
        full["new"] = None
    if case["what"] == "round" and case["path"] == "call":
        full["deleted"] = None
    return full
