"""K-column calls: how finely FP32 products are folded into the compensated sums, and the memory a call takes."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2404_08299_gb300 import build
    build.build()
    torch.cuda.init()


def prdf():
    import paper_2404_08299_gb300 as p
    return p


@pytest.mark.parametrize("K", [1, 2, 4, 8, 16, 32, 64])
@pytest.mark.parametrize("deg", [8, 16, 97, 128, 200])
def test_fp32_products_are_folded_by_fours(deg, K):
    """A row of terms 1, q, q, q, ... with q = 0.4 ulp(1): added one by one to 1 in FP32 every q is lost, so of a block
    of b products that starts with the 1, (b - 1) q are. Blocks of four lose at most 3 q where the row's edges lie in
    order (rows by slots) or strided by slots (chunks: the slot with the 1 loses 3 q); the compensated sum keeps the
    rest, and its rounding adds half an ulp. The sum is read back exactly through an edge to a further vertex (alpha =
    1/2, one edge a source, so every product is exact)."""
    q = 0.4 * 2.0 ** -23
    n = deg + 2
    v, x = deg, deg + 1
    src = torch.arange(deg + 1, dtype=torch.int32, device="cuda")
    dst = torch.full((deg + 1,), v, dtype=torch.int32, device="cuda")
    dst[deg] = x
    g = prdf().Graph(n, src, dst, torch.ones(deg + 1, device="cuda"), self_loops=False)
    term = np.full(deg, np.float32(q), np.float64)
    term[0] = 1.0
    S = torch.zeros(n, K, dtype=torch.float64, device="cuda")
    S[:deg] = 2 * torch.from_numpy(term).cuda()[:, None]  # a source's rank is S / 2
    R, st = g.pagerank_ppr(S, alpha=0.5, precision=1, tol=10.0, tol_fp32_rel=1e-9)
    assert st.iterations - st.iterations_fp32 == 1
    got = 4 * R[x]  # R[x] = R32[v] / 2, R32[v] = sum / 2
    err = (got - term.sum()).abs().max().item() / 2.0 ** -23
    lost = 3 * 0.4
    assert err <= lost + 0.5 + deg * 2.0 ** -23


def test_memory_of_a_call_without_long_rows():
    """Rows of at most 90 entries, so no chunks of long rows: an FP64 call takes the state (24 bytes a vertex and column)
    and its tables (16 bytes a vertex, 4 more a vertex and tile of 64 columns), and no room for partial sums of chunks.
    64 MB are left for the pool's granularity."""
    n, deg, K = 20000, 90, 2048
    gen = torch.Generator(device="cuda").manual_seed(3)
    i = torch.arange(n, device="cuda")
    src = torch.cat([(i + int(k)) % n for k in torch.randperm(n - 1, device="cuda", generator=gen)[:deg - 1] + 1])
    g = prdf().Graph(n, src.int(), i.repeat(deg - 1).int(), torch.ones(src.numel(), device="cuda"))
    S = torch.rand(n, K, dtype=torch.float64, device="cuda", generator=gen)
    g.pagerank_ppr(S[:, :3].contiguous(), max_iter=2)
    R = torch.empty(n, K, dtype=torch.float64, device="cuda")
    del R  # (the result's memory is there: torch hands the block out again)
    prdf().release_cached_memory()
    before = torch.cuda.mem_get_info()[0]
    R, _ = g.pagerank_ppr(S, max_iter=2)
    prdf().release_cached_memory()
    used = before - torch.cuda.mem_get_info()[0]
    assert used <= 24 * n * K + 16 * n + 4 * n * (K // 64) + (64 << 20), used
