"""The rank loop's work units at the sizes where they can go wrong: vertex counts around a warp, a batch and a unit
of rows, rows around every class bound and around the hub chunk, and frontier rows of more than one list entry.
Tolerances are those of the other parity tests: Static takes the oracle's sweep count and lies within 1e-13 (the
same iteration, rounding-level differences), DF-P flags are exact and ranks lie within 1e-12 relative."""
import numpy as np
import pytest
import torch

import oracle
from helpers import batch_case, dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2404_08299_gb300 import build
    build.build()
    torch.cuda.init()


def row_lengths_graph(n, degrees, seed):
    """Vertex v < len(degrees) has exactly degrees[v] in-edges with its self-loop; the others a few."""
    rng = np.random.default_rng(seed)
    s, d = [], []
    for v, k in enumerate(degrees):
        others = np.delete(np.arange(n, dtype=np.int32), v)
        s.append(rng.choice(others, k - 1, replace=False).astype(np.int32))
        d.append(np.full(k - 1, v, np.int32))
    return n, np.concatenate(s), np.concatenate(d)


BOUNDS = [1, 2, 3, 4, 5, 8, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 513, 1023, 1024,
          1025, 2049, 4095, 4096, 4097, 5119, 5120, 5121]


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 65, 255, 256, 257, 511, 513, 1025])
def test_vertex_counts_around_a_unit(n):
    import paper_2404_08299_gb300 as prdf
    rng = np.random.default_rng(n)
    s, d = (rng.integers(0, n, 6 * n).astype(np.int32) for _ in range(2))
    g = prdf.Graph(n, dev(s), dev(d))
    Ro, sto = oracle.pagerank_static(oracle.graph(n, s, d))
    for precision in (0, 1):
        R, st = g.pagerank_static(precision=precision)
        assert st.converged
        if precision == 0:
            assert st.iterations == sto.iterations
            assert np.max(np.abs(host(R) - Ro)) <= 1e-13
        else:
            assert np.max(np.abs(host(R) - Ro)) <= 1e-8


@pytest.mark.parametrize("copies", [1, 3])
def test_row_lengths_around_the_class_bounds(copies):
    import paper_2404_08299_gb300 as prdf
    n, s, d = row_lengths_graph(6000, BOUNDS * copies, seed=copies)
    g = prdf.Graph(n, dev(s), dev(d))
    Ro, sto = oracle.pagerank_static(oracle.graph(n, s, d))
    R, st = g.pagerank_static()
    assert st.iterations == sto.iterations and np.max(np.abs(host(R) - Ro)) <= 1e-13
    Rh, sth = g.pagerank_static(time_sweeps=1, check_every=3)
    assert torch.equal(R, Rh) and sth.iterations == st.iterations


@pytest.mark.parametrize("reverse", [False, True])
@pytest.mark.parametrize("size", [1, 40, 400])
def test_dfp_with_long_rows(reverse, size):
    """Rows of every length as in-rows (hub chunks) or out-rows (frontier entries of 1024 edges)."""
    n, s, d = row_lengths_graph(6000, BOUNDS, seed=7)
    if reverse:
        s, d = d, s
    hubs = np.arange(len(BOUNDS), dtype=np.int32)
    ins = (hubs, hubs[::-1].copy()) if reverse else (np.arange(3000, 3000 + len(hubs), dtype=np.int32), hubs)
    empty = np.zeros(0, np.int32)
    g, og1, R0, (ds, dd, is_, id_, de, ie, dmo, imo) = batch_case(n, s, d, 3, size, extra=(empty, empty, *ins))
    for kw in ({}, {"expand_pull": 0.0}, {"expand_pull": 1.0}, {"prune": 0}):
        R, st, dV = g.pagerank_dfp(dev(ds), dev(dd), dev(is_), R0, del_mask=de, ins_mask=ie, want_dV=True, **kw)
        Ro, sto, dVo, _ = oracle.pagerank_dfp(og1, ds, dd, is_, host(R0), del_mask=dmo, ins_mask=imo,
                                              prune=bool(kw.get("prune", 1)))
        assert st.iterations == sto.iterations
        assert np.max(np.abs(host(R) - Ro) / Ro) <= 1e-12
        assert np.array_equal(host(dV), dVo)


@pytest.mark.parametrize("n", [18225, 1001, 1002, 1003, 4097])
def test_dfp_flags_at_the_end_of_the_numbering(n):
    """Short rows only, so the scan's last word of flags ends inside its padding; memory that other graphs used
    before, so the padding is not zero by chance. Flags and sweep count are the oracle's, and ranks of vertices
    that were never affected are untouched."""
    for _ in range(3):
        m = 40000
        s, d = (np.random.default_rng(m).integers(0, m, 8 * m).astype(np.int32) for _ in range(2))
        dynamic = batch_case(m, s, d, 1, 400)
        del dynamic
    v = np.arange(n, dtype=np.int32)
    s = np.concatenate([v, (v + 1) % n, v, (v + 7) % n])
    d = np.concatenate([(v + 1) % n, v, (v + 7) % n, v])
    g, og1, R0, (ds, dd, is_, id_, de, ie, dmo, imo) = batch_case(n, s, d, n, 3)
    R, st, dV = g.pagerank_dfp(dev(ds), dev(dd), dev(is_), R0, del_mask=de, ins_mask=ie, want_dV=True, prune=0)
    Ro, sto, dVo, _ = oracle.pagerank_dfp(og1, ds, dd, is_, host(R0), del_mask=dmo, ins_mask=imo, prune=False)
    assert st.iterations == sto.iterations and np.array_equal(host(dV), dVo)
    assert np.max(np.abs(host(R) - Ro) / Ro) <= 1e-12
