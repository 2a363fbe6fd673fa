"""The K-column loop's work units and the weighted graph's layouts at the sizes where they can go wrong: rows around
the bound of the long rows and around every chunk size, column counts around a tile, graphs on both sides of the chunk
rule's edge counts, weights on every form of the radix build, and new weights between batches. Solves lie within 1e-8
of the oracle (the library's tolerance, as in the other parity tests); ids and weights are exact."""
import numpy as np
import pytest
import torch

import oracle
import synth
from helpers import dev, host
from test_gpu_sweep_units import row_lengths_graph

pytestmark = pytest.mark.gpu

ROWS = [2, 3, 4, 5, 7, 8, 9, 31, 32, 33, 47, 48, 49, 50, 95, 96, 97, 98, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025,
        2047, 2048, 2049]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2404_08299_gb300 import build
    build.build()
    torch.cuda.init()


def prdf():
    import paper_2404_08299_gb300 as p
    return p


def with_weights(n, s, d, seed):
    """The graph with a self-loop and a weight on every vertex, the oracle's graph and its weights."""
    loops = np.arange(n, dtype=np.int32)
    s2, d2 = np.concatenate([s, loops]), np.concatenate([d, loops])
    g = prdf().Graph(n, dev(s2), dev(d2), dev(synth.edge_weights(s2, d2, seed=seed)))
    og = oracle.graph(n, s2, d2)
    rows, cols = oracle.csr_to_edges(og.out_off, og.out_adj)
    return g, og, synth.edge_weights(rows, cols, seed=seed).astype(np.float64)


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("reverse", [False, True])
@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 8, 9, 16, 17, 32, 33, 64, 65])
def test_rows_and_columns_around_a_unit(K, reverse, precision):
    n, s, d = row_lengths_graph(2100, ROWS, seed=K)
    if reverse:  # the long rows are the adjoint's
        s, d = d, s
    g, og, w = with_weights(n, s, d, seed=K)
    S = synth.ppr_seeds(n, K, n_seed=16, seed=K + 1)
    G = synth.normal((n, K), seed=K + 2)
    R, st = g.pagerank_ppr(dev(S), precision=precision)
    gS, gw, stb = g.pagerank_backward(R, dev(G), precision=precision)
    P = oracle.row_normalise(og, w)
    Ro, _ = oracle.ppr(og, P, S, tol=1e-15, max_iter=1000)
    _, gSo, gwo, _ = oracle.ppr_adjoint(og, w, P, Ro, G, tol=1e-15, max_iter=1000)
    assert st.converged and stb.converged
    assert np.max(np.abs(host(R) - Ro)) <= 1e-8
    assert np.max(np.abs(host(gS) - gSo)) <= 1e-8 * max(1.0, np.abs(gSo).max())
    assert np.max(np.abs(host(gw) - gwo)) <= 1e-8 * max(1.0, np.abs(gwo).max())


@pytest.mark.parametrize("n,K", [(1, 3), (2, 5), (31, 2), (33, 17), (257, 7)])
def test_few_vertices(n, K):
    rng = np.random.default_rng(n)
    s, d = (rng.integers(0, n, 6 * n).astype(np.int32) for _ in range(2))
    g, og, w = with_weights(n, s, d, seed=n)
    S = synth.uniform((n, K), seed=n) + 0.01
    S /= S.sum(axis=0, keepdims=True)
    Ro, _ = oracle.ppr(og, oracle.row_normalise(og, w), S, tol=1e-15, max_iter=1000)
    for precision in (1, 0):
        R, st = g.pagerank_ppr(dev(S), precision=precision)
        assert st.converged and np.max(np.abs(host(R) - Ro)) <= 1e-8


@pytest.mark.parametrize("nsamp", [3 << 20, 3 << 21, 9 << 22])
def test_chunk_rules_on_larger_graphs(nsamp):
    """Edge counts on both sides of 2^22 and of 2^25, against 200 power iterations (0.85^200 < 1e-14) by a sparse
    product in FP64; the library's weights are read back, so the two share the transition matrix only."""
    n, s, d = synth.rmat(20, nsamp, seed=5)
    g = prdf().Graph(n, dev(s), dev(d), dev(synth.edge_weights(s, d, seed=5)))
    off, adj, w = g.export_csr(prdf().PRDF_IN)
    src = adj.long()
    tot = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, src, w.double())
    A = torch.sparse_csr_tensor(off, src, w.double() / tot[src], size=(n, n))
    S = dev(synth.ppr_seeds(n, 5, n_seed=16, seed=6))
    X = S.clone()
    for _ in range(200):
        X = 0.85 * (A @ X) + 0.15 * S
    R, st = g.pagerank_ppr(S)
    assert st.converged and float((R - X).abs().max()) <= 1e-8


@pytest.mark.parametrize("n,m0", [(3, 1), (1000, 3096), (1000, 3097), (70001, 500000), ((1 << 17) + 3, 1 << 20),
                                  ((1 << 20) + 5, 3000)])
@pytest.mark.parametrize("self_loops", [True, False])
def test_weighted_radix_build(n, m0, self_loops):
    """Weighted lists at the sizes of the unweighted radix test: duplicates keep their largest weight, given
    self-loops theirs, and missing ones weigh 1."""
    rng = np.random.default_rng(n + m0)
    s = (rng.integers(0, n, m0) if n < 1000 else rng.zipf(1.3, m0) % n).astype(np.int64)
    d = rng.integers(0, n, m0).astype(np.int64)
    d[::7] = s[::7]
    w = rng.uniform(0.5, 1.5, m0).astype(np.float32)
    g = prdf().Graph(n, dev(s.astype(np.int32)), dev(d.astype(np.int32)), dev(w), self_loops=self_loops)
    v = np.arange(n, dtype=np.int64)
    for which, (r, c) in ((prdf().PRDF_OUT, (s, d)), (prdf().PRDF_IN, (d, s))):
        key, inv = np.unique(r * n + c, return_inverse=True)
        best = np.zeros(len(key), np.float32)
        np.maximum.at(best, inv, w)
        if self_loops:
            miss = np.setdiff1d(v * n + v, key)
            key, best = np.concatenate([key, miss]), np.concatenate([best, np.ones(len(miss), np.float32)])
            order = np.argsort(key)
            key, best = key[order], best[order]
        off, adj, wg = (host(x) for x in g.export_csr(which))
        assert np.array_equal(off, np.searchsorted(key, np.arange(n + 1) * n))
        assert np.array_equal(adj, key % n) and np.array_equal(wg, best)


def test_new_weights_between_batches():
    """New weights on a numbered graph, twice, then a small batch (which shifts the slots) and new weights again:
    each time the graph answers as one made with those weights, on both CSRs and in a solve."""
    n, s, d = synth.rmat(11, 20000, seed=31)
    g, og, _ = with_weights(n, s, d, seed=31)
    S = dev(synth.ppr_seeds(n, 6, n_seed=16, seed=32))
    for step in range(4):
        if step == 2:
            ds, dd, is_, id_ = synth.batch(n, og.out_off, og.out_adj, 40, seed=33, s1=1)
            g.apply_batch(dev(ds), dev(dd), dev(is_), dev(id_), ins_w=torch.ones(len(is_), device="cuda"))
            og, _, _ = oracle.apply_batch(og, ds, dd, is_, id_)
        rows, cols = oracle.csr_to_edges(og.out_off, og.out_adj)
        w = synth.edge_weights(rows, cols, seed=40 + step)
        g.set_weights(dev(w))
        fresh = prdf().Graph(n, dev(rows), dev(cols), dev(w))
        for which in (prdf().PRDF_OUT, prdf().PRDF_IN):
            for a, b in zip(g.export_csr(which), fresh.export_csr(which)):
                assert torch.equal(a, b)
        R, _ = g.pagerank_ppr(S)
        Ro, _ = oracle.ppr(og, oracle.row_normalise(og, w.astype(np.float64)), host(S), tol=1e-15, max_iter=1000)
        assert np.max(np.abs(host(R) - Ro)) <= 1e-8


@pytest.mark.parametrize("nd,ni", [(0, 1), (1, 0), (1, 4096), (4096, 1), (4096, 4096), (4096, 4097), (4097, 0)])
def test_batches_around_the_one_block_bound(nd, ni):
    """Deletions and insertions on both sides of the preparation in one block, lists of unequal length, every
    entry on a few rows."""
    n, s, d = synth.rmat(15, 1 << 19, seed=41)
    g = prdf().Graph(n, dev(s), dev(d))
    og = oracle.graph(n, s, d)
    rng = np.random.default_rng(nd + ni)
    rows, cols = oracle.csr_to_edges(og.out_off, og.out_adj)
    pick = rng.choice(og.m, nd, replace=False)
    ds, dd = rows[pick].astype(np.int32), cols[pick].astype(np.int32)
    is_, id_ = rng.integers(0, 40, ni).astype(np.int32), rng.integers(0, n, ni).astype(np.int32)
    de, ie = g.apply_batch(dev(ds), dev(dd), dev(is_), dev(id_))
    og, dmo, imo = oracle.apply_batch(og, ds, dd, is_, id_)
    assert np.array_equal(host(de), dmo) and np.array_equal(host(ie), imo)
    for which, o, a in ((prdf().PRDF_OUT, og.out_off, og.out_adj), (prdf().PRDF_IN, og.in_off, og.in_adj)):
        off, adj, _ = g.export_csr(which)
        assert np.array_equal(host(off), o) and np.array_equal(host(adj), a)
