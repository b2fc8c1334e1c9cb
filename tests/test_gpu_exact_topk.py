"""Exact search and the FP32 PartialReduce on small integers: every FP32 score
is exact and most of them tie, so values and indices (larger score first, then
the smaller row) are decided exactly, at the edges of the selection's blocks of
8192 scores, of its K limits and of the FP32 kernel's tiles."""
import pytest
import torch

from paper_2206_14286_gb300 import search as S
from tests.gpu_util import ensure_built

pytestmark = pytest.mark.gpu


def rows(n, D, seed, lo=-3, hi=4):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randint(lo, hi, (n, D), generator=g, device="cuda").float()


def ranked(s, K):
    """(values, columns) of the best K per row, ties to the smaller column."""
    o = torch.sort(s, dim=1, descending=True, stable=True)
    return o.values[:, :K], o.indices[:, :K]


@pytest.mark.parametrize("dtype,metric", [("f32", "ip"), ("f32", "l2"), ("bf16", "ip")])
@pytest.mark.parametrize("N,K", [(5, 1), (5, 5), (100, 33), (8191, 10), (8192, 128), (8193, 129),
                                 (8200, 8192 // 8), (20_000, 31), (20_000, 32), (20_000, 1024),
                                 (20_000, 1025), (200_001, 100)])
def test_exact_search_order(dtype, metric, N, K):
    ensure_built()
    for M in (1, 70):
        x, q = rows(N, 20, N + K), rows(M, 20, 7 * N + K)
        d = S.Database(x, metric=metric, dtype=dtype)
        val, idx = d.search_exact(q, K)
        s = (q.double() @ x.double().t())
        if metric == "l2":
            s = -((q * q).double().sum(1)[:, None] + (x * x).double().sum(1)[None, :] - 2.0 * s)
        v, a = ranked(s, K)
        assert torch.equal(idx.long(), a)
        assert torch.equal(val.double(), -v if metric == "l2" else v)


def test_exact_search_all_equal_and_many_chunks():
    """Every score ties (more elements at the bound than its buffer holds),
    and enough queries that the rows come in many chunks."""
    ensure_built()
    x = torch.ones((30_000, 16), device="cuda")
    for M, K in ((3, 10), (3, 200), (2000, 40)):
        q = rows(M, 16, M)
        d = S.Database(x, metric="ip", dtype="f32")
        val, idx = d.search_exact(q, K)
        assert torch.equal(idx, torch.arange(K, device="cuda", dtype=torch.int32).expand(M, K))
        assert torch.equal(val, q.sum(1, keepdim=True).expand(M, K))


def test_exact_search_skips_infinities_and_nan():
    ensure_built()
    x, q = rows(9000, 16, 1), rows(5, 16, 2, 1, 3)
    x[10] = -float("inf")
    x[20, 3] = float("nan")
    x[8999] = float("inf")
    d = S.Database(x, metric="ip", dtype="f32")
    _, idx = d.search_exact(q, 50)
    assert (idx[:, 0] == 8999).all()
    assert not ((idx == 10) | (idx == 20)).any()


@pytest.mark.parametrize("M", [1, 63, 64, 65, 127, 128, 129, 300])
@pytest.mark.parametrize("N,L", [(1, 1), (63, 5), (64, 64), (5003, 5), (5003, 65), (5003, 5003),
                                 (40_000, 1000)])
def test_partial_reduce_f32_order(M, N, L):
    """Bins (folded when L < 64), splits of the rows merged by 64-bit keys."""
    ensure_built()
    x, q = rows(N, 24, N + L), rows(M, 24, M)
    d = S.Database(x, metric="ip", dtype="f32")
    V, A = d.partial_reduce(q, L)
    s = (q @ x.t()).double()
    T = -(-N // L)
    p = torch.full((M, T * L), -1e30, dtype=torch.float64, device="cuda")
    p[:, :N] = s
    p = p.view(M, T, L)
    best = p.amax(1)
    first = (p == best[:, None, :]).to(torch.uint8).argmax(1) * L + torch.arange(L, device="cuda")
    assert torch.equal(V.double(), best)
    assert torch.equal(A.long(), first)


@pytest.mark.parametrize("M,N", [(65, 9728), (65, 9729), (333, 3000), (333, 3300), (1000, 1216),
                                 (1000, 1217), (129, 100), (4865, 65), (9729, 65)])
def test_exact_search_tile_sizes(M, N):
    """FP32 tiles of 128 rows, or of 64 where the larger would leave half of the
    SMs without one."""
    ensure_built()
    x, q = rows(N, 20, M), rows(M, 20, N)
    d = S.Database(x, metric="ip", dtype="f32")
    val, idx = d.search_exact(q, 10)
    v, a = ranked(q @ x.t(), 10)
    assert torch.equal(idx.long(), a)
    assert torch.equal(val, v)


def test_exact_search_of_few_rows_is_shared_out():
    """128 queries on 3000 long rows, in tiles of 128 x 64, take up to 1.65 times
    as long as 64 in tiles of 64 x 64 (with 24 tiles of 128 x 128, twice)."""
    ensure_built()
    x, q = rows(3000, 4096, 1), rows(128, 4096, 2)
    d = S.Database(x, metric="ip", dtype="f32")

    def us(q):
        for _ in range(3):
            d.search_exact(q, 10)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t = []
        for _ in range(9):
            a.record()
            for _ in range(4):
                d.search_exact(q, 10)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        return min(t)

    assert us(q) < 1.65 * us(q[:64])
