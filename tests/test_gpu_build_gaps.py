"""Builds whose edges sit on few vertices: the offsets of long runs of empty rows (a run a lane, a warp or the whole GPU
writes), on both CSRs, against a count in numpy, and the time they take."""
import time

import numpy as np
import pytest
import torch

from helpers import dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2404_08299_gb300 import build
    build.build()
    torch.cuda.init()


def prdf():
    import paper_2404_08299_gb300 as p
    return p


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("used", ["low", "high", "both", "steps", "one"])
@pytest.mark.parametrize("n,m0", [(1001, 512), (65535, 8192), (65537, 4096), (65600, 5000), ((1 << 18) + 3, 1 << 15),
                                  ((1 << 20) + 5, 70001)])
def test_offsets_of_empty_rows(n, m0, used, weighted):
    rng = np.random.default_rng(n + m0)
    ids = {"low": np.arange(min(n, 300)), "high": np.arange(n - 300, n), "one": np.array([n // 2]),
           "both": np.concatenate([np.arange(100), np.arange(n - 100, n)]),
           # runs of 63 to 66 rows and of 65535 to 65537 between used ones
           "steps": np.cumsum(np.tile([1, 63, 64, 65, 66, 67], 4 if n < 2000 else 30))}[used]
    if used == "steps" and n > 1 << 18:
        ids = np.concatenate([ids, ids[-1] + np.cumsum([65535, 65536, 65537])])
    ids = ids[ids < n]
    s, d = ids[rng.integers(0, len(ids), m0)].astype(np.int64), ids[rng.integers(0, len(ids), m0)].astype(np.int64)
    w = rng.uniform(0.5, 1.5, m0).astype(np.float32)
    g = prdf().Graph(n, dev(s.astype(np.int32)), dev(d.astype(np.int32)), dev(w) if weighted else None,
                     self_loops=False)
    for which, (r, c) in ((prdf().PRDF_OUT, (s, d)), (prdf().PRDF_IN, (d, s))):
        key, inv = np.unique(r * n + c, return_inverse=True)
        off, adj, wg = g.export_csr(which)
        assert np.array_equal(host(off), np.searchsorted(key, np.arange(n + 1) * n))
        assert np.array_equal(host(adj), key % n)
        if weighted:
            best = np.zeros(len(key), np.float32)
            np.maximum.at(best, inv, w)
            assert np.array_equal(host(wg), best)


@pytest.mark.parametrize("weighted", [False, True])
def test_time_does_not_depend_on_where_the_rows_are(weighted):
    """16.8 M vertices, 1 M edges on the first 32,768 ids or spread over all: the passes are the same, so the builds take
    about as long (within three times; a lane that wrote every offset after the last used row took 45 times)."""
    n, m0 = 1 << 24, 1 << 20
    gen = torch.Generator(device="cuda").manual_seed(1)
    w = torch.rand(m0, device="cuda", generator=gen) + 0.5 if weighted else None
    ms = []
    for top in (n, n >> 9):
        s, d = (torch.randint(top, (m0,), device="cuda", generator=gen, dtype=torch.int32) for _ in range(2))
        best = 1e9
        for _ in range(4):
            torch.cuda.synchronize()
            t = time.perf_counter()
            g = prdf().Graph(n, s, d, w, self_loops=False)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
            del g
        ms.append(1e3 * best)
    assert ms[1] <= 3 * ms[0], ms
