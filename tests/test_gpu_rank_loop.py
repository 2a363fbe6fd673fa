"""The rank loop on graphs of more than 6.3 M in-edges, where rows of 129 to 4096 entries are a warp each and longer ones
go by four 1024-edge chunks a unit, loops that max_iter cuts off, out-degrees that a float does not hold, and sums that
depend on their order. Flags, counts and sweep numbers are the oracle's; ranks lie within 1e-12 relative of it (the
same iteration, rounding-level differences), as in the other parity tests."""
import numpy as np
import pytest
import torch

import oracle
import synth
from helpers import batch_case, dev, dynamic_case, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2404_08299_gb300 import build
    build.build()
    torch.cuda.init()


def prdf():
    import paper_2404_08299_gb300 as p
    return p


PLANTED = [129, 130, 255, 257, 511, 512, 513, 514, 1023, 1024, 1025, 1026, 2047, 2048, 2049, 2050, 4095, 4096, 4097,
           4099, 5000, 5121, 6000, 7169, 9000, 12000, 16385, 20000, 30000, 40000]


@pytest.fixture(scope="module")
def large():
    """More than 6.3 M in-edges, so rows of 129 to 4096 are a warp each and longer ones go by four 1024-edge chunks a
    unit; vertex k < len(PLANTED) has about PLANTED[k] in-edges, and a batch adds one to each."""
    n, s, d = synth.rmat(18, 1 << 23, seed=71)
    keep = d >= len(PLANTED)
    s, d = s[keep], d[keep]
    rng = np.random.default_rng(71)
    hs = [rng.choice(np.arange(len(PLANTED), n - 100, dtype=np.int32), k, replace=False) for k in PLANTED]
    hd = [np.full(k, v, np.int32) for v, k in enumerate(PLANTED)]
    s, d = np.concatenate([s, *hs]).astype(np.int32), np.concatenate([d, *hd]).astype(np.int32)
    empty = np.zeros(0, np.int32)
    ins = (np.arange(n - len(PLANTED), n, dtype=np.int32), np.arange(len(PLANTED), dtype=np.int32))
    case = batch_case(n, s, d, 72, 60, extra=(empty, empty, *ins))
    assert case[1].m > 6 << 20 and (case[1].indeg > 4096).sum() >= 10
    return case


@pytest.mark.parametrize("kw", [{}, {"prune": 0}, {"expand_pull": 0.0}, {"expand_pull": 2.0}])
def test_dfp_with_rows_of_several_chunks(large, kw):
    g, og1, R0, (ds, dd, is_, id_, de, ie, dmo, imo) = large
    args = dev(ds), dev(dd), dev(is_), R0
    R, st, dV = g.pagerank_dfp(*args, del_mask=de, ins_mask=ie, want_dV=True, **kw)
    Ro, sto, dVo, trace = oracle.pagerank_dfp(og1, ds, dd, is_, host(R0), del_mask=dmo, ins_mask=imo,
                                              prune=bool(kw.get("prune", 1)))
    assert st.affected_initial == trace[0]
    assert st.iterations == sto.iterations and np.array_equal(host(dV), dVo)
    assert np.max(np.abs(host(R) - Ro) / Ro) <= 1e-12
    Rh, sth, dVh = g.pagerank_dfp(*args, del_mask=de, ins_mask=ie, want_dV=True, time_sweeps=1, check_every=3, **kw)
    assert torch.equal(R, Rh) and torch.equal(dV, dVh) and sth.affected_initial == trace[0]


def test_static_and_dt_with_rows_of_several_chunks(large):
    g, og1, R0, (ds, dd, is_, id_, de, ie, dmo, imo) = large
    R, st = g.pagerank_static()
    Ro, sto = oracle.pagerank_static(og1)
    assert st.iterations == sto.iterations and np.max(np.abs(host(R) - Ro) / Ro) <= 1e-12
    R, st, dV = g.pagerank_dt(dev(ds), dev(dd), dev(is_), R0, del_mask=de, ins_mask=ie, want_dV=True)
    Ro, sto, dVo, na, _ = oracle.pagerank_dt(og1, ds, dd, is_, host(R0), del_mask=dmo, ins_mask=imo)
    assert st.affected_initial == na and st.iterations == sto.iterations and np.array_equal(host(dV), dVo)
    assert np.max(np.abs(host(R) - Ro) / Ro) <= 1e-12


@pytest.mark.parametrize("expand_pull", [0.0, 2.0])
@pytest.mark.parametrize("max_iter", [1, 2, 3, 5])
@pytest.mark.parametrize("prune", [1, 0])
def test_dfp_stopped_by_max_iter(prune, max_iter, expand_pull):
    """The affected set after a sweep that did not converge includes that sweep's expansion, the last one's too
    (Alg. frontier), and the mixed solve's FP64 stage starts from it."""
    g, og1, R0, (ds, dd, is_, id_, de, ie, dmo, imo) = dynamic_case(5, 12, 40000, 4)
    kw = dict(del_mask=de, ins_mask=ie, want_dV=True, prune=prune, max_iter=max_iter, expand_pull=expand_pull)
    args = dev(ds), dev(dd), dev(is_), R0
    R, st, dV = g.pagerank_dfp(*args, **kw)
    Ro, sto, dVo, _ = oracle.pagerank_dfp(og1, ds, dd, is_, host(R0), del_mask=dmo, ins_mask=imo, prune=bool(prune),
                                          max_iter=max_iter)
    assert not sto.converged and st.iterations == sto.iterations == max_iter
    assert np.array_equal(host(dV), dVo)
    assert np.max(np.abs(host(R) - Ro) / Ro) <= 1e-12
    for precision in (0, 1):
        (R, st, dV), (Rh, sth, dVh) = (g.pagerank_dfp(*args, precision=precision, time_sweeps=t, **kw) for t in (0, 1))
        assert torch.equal(dV, dVh) and torch.equal(R, Rh)


@pytest.mark.parametrize("above", [1, 1025])
def test_fp32_frontier_of_an_out_degree_past_a_floats_integers(above):
    """A vertex with 2^24 + above out-edges (its self-loop included), above = 1 modulo 1024, joins the frontier in an
    FP32 sweep: every out-neighbour is marked, the last one too (DF keeps every mark)."""
    n = (1 << 24) + above
    hub = torch.zeros(n - 1, dtype=torch.int32, device="cuda")
    g = prdf().Graph(n, hub, torch.arange(1, n, dtype=torch.int32, device="cuda"))
    R0, _ = g.pagerank_static(max_iter=3)
    e = torch.zeros(0, dtype=torch.int32, device="cuda")
    one = torch.ones(1, dtype=torch.int32, device="cuda")
    de, ie = g.apply_batch(e, e, one, torch.zeros_like(one))  # 1 -> hub
    R, st, dV = g.pagerank_dfp(e, e, one, R0, ins_mask=ie, want_dV=True, prune=0, precision=1, expand_pull=2.0,
                               max_iter=8)
    assert int(dV.sum()) == n


def random_rows(n, lo, hi, seed):
    """lo to hi in-edges a vertex from random sources."""
    rng = np.random.default_rng(seed)
    d = np.repeat(np.arange(n, dtype=np.int32), rng.integers(lo, hi + 1, n))
    return n, rng.integers(0, n, len(d)).astype(np.int32), d


@pytest.mark.parametrize("call", ["pagerank_dfp", "pagerank_dt"])
@pytest.mark.parametrize("kw", [{"precision": 1}, {"accumulate": 1}, {"accumulate": 1, "prune": 0}])
@pytest.mark.parametrize("graph", ["rows", "rmat"])
def test_every_run_gives_the_same_bits(graph, kw, call):
    """FP32 sums and plain FP64 sums round by the order of their terms. The affected rows are listed in an order that
    changes from run to run, so rows of 5 to 32 entries come in batches of every size."""
    case = batch_case(*random_rows(100003, 8, 15, 1), 3, 300) if graph == "rows" else dynamic_case(9, 20, 1 << 24, 300)
    g, og1, R0, (ds, dd, is_, id_, de, ie, dmo, imo) = case
    out = [getattr(g, call)(dev(ds), dev(dd), dev(is_), R0, del_mask=de, ins_mask=ie, want_dV=True,
                            time_sweeps=int(k % 3 == 2), **kw) for k in range(9)]
    R, st, dV = out[0]
    for Rk, stk, dVk in out[1:]:
        assert torch.equal(R, Rk) and torch.equal(dV, dVk)
        assert st.iterations == stk.iterations and st.iterations_fp32 == stk.iterations_fp32


@pytest.mark.parametrize("old", [1, 2, 6, 20, 60])
def test_a_row_that_outgrew_its_class(old):
    """A vertex of `old` in-edges gains 100,000 in a batch that keeps the numbering. Its row is walked by as many lanes
    as in the class of a warp per row, so a solve takes no longer than twice that of a graph built with the row there
    (the rest of a sweep is the same; a lane or a few of them alone take up to fifty times as long), in Static and in
    DF, whose ranks and flags are those of the fresh graph."""
    n, s, d = synth.rmat(19, 1 << 23, seed=81)
    keep = d != 5
    s, d = s[keep], d[keep]
    src = np.arange(n - 200000, n, dtype=np.int32)
    s = np.concatenate([s, src[:old - 1]]).astype(np.int32)
    d = np.concatenate([d, np.full(old - 1, 5, np.int32)]).astype(np.int32)
    g = prdf().Graph(n, dev(s), dev(d))
    new = dev(src[1000:101000])
    e = torch.zeros(0, dtype=torch.int32, device="cuda")
    g.apply_batch(e, e, new, torch.full_like(new, 5))
    assert g.m > 6 << 20
    fresh = prdf().Graph(n, torch.cat([dev(s), new]), torch.cat([dev(d), torch.full_like(new, 5)]))
    fresh.set_thresholds(prdf().PRDF_IN, [1, 4, 16, 32, 128, 1 << 30])
    assert fresh.m == g.m
    ms = {}
    for name, x in (("grown", g), ("fresh", fresh)):
        for precision in (0, 1):
            x.pagerank_static(precision=precision)
            ms[name, precision] = min(x.pagerank_static(precision=precision)[1].ms_iterate for _ in range(3))
    Rg, stg = g.pagerank_static()
    Rf, stf = fresh.pagerank_static()
    assert torch.equal(Rg, Rf) and stg.iterations == stf.iterations
    for precision in (0, 1):
        assert ms["grown", precision] <= 2 * ms["fresh", precision]
    (Rg, stg, dVg), (Rf, stf, dVf) = (x.pagerank_dfp(e, e, new, Rf, want_dV=True, prune=0, tol=1e-14, tau_f=1e-9)
                                      for x in (g, fresh))
    assert torch.equal(Rg, Rf) and torch.equal(dVg, dVf) and stg.iterations == stf.iterations
    assert stg.affected_initial == stf.affected_initial
