"""The approx_max_k / approx_min_k operator on a given score matrix against
the FP64 oracle: bit-exact values (the inputs are FP32 or BF16 numbers) and
indices, for both bin maps, with and without aggregation to top-K."""
import numpy as np
import pytest
import torch

import oracle
from paper_2206_14286_gb300 import search as S
from tests.gpu_util import ensure_built

pytestmark = pytest.mark.gpu


def scores(M, N, seed, ties=True):
    g = np.random.Generator(np.random.PCG64(seed))
    X = g.standard_normal((M, N)).astype(np.float32)
    if ties:
        # repeated values and zeros of both signs exercise the tie rule
        X[:, ::7] = np.round(X[:, ::7])
        X[:, 3::11] = -0.0
    return X


@pytest.mark.parametrize("bins", ["mod", "contiguous"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_approx_max_k_matches_oracle(bins, dtype):
    ensure_built()
    M, N, K = 37, 5003, 10
    X = scores(M, N, 41)
    t = torch.from_numpy(X).cuda()
    if dtype == "bf16":
        t = t.to(torch.bfloat16)
    Xo = t.float().cpu().numpy().astype(np.float64)
    for L in (1, 7, 128, 1000, N):
        for is_min in (False, True):
            for agg in (False, True):
                k = min(K, L)
                v, i = S.approx_max_k(t, k, L=L, bins=bins, is_min=is_min, aggregate_to_topk=agg)
                ov, oi = oracle.approx_max_k(Xo, k, L, bins=bins, is_min=is_min,
                                             aggregate_to_topk=agg)
                v, i = v.cpu().numpy(), i.cpu().numpy()
                assert np.array_equal(i, oi), (L, is_min, agg)
                assert np.array_equal(v.astype(np.float64), ov), (L, is_min, agg)


def test_approx_max_k_many_rows_and_planned_bins():
    ensure_built()
    M, N, K = 70000, 64, 4                      # more rows than one grid dimension holds
    X = scores(M, N, 42)
    t = torch.from_numpy(X).cuda()
    v, i = S.approx_max_k(t, K, L=8)
    ov, oi = oracle.approx_max_k(X.astype(np.float64), K, 8)
    assert np.array_equal(i.cpu().numpy(), oi)
    # L from the recall law, and from a larger planning size (a shard of a
    # bigger input): the output width follows the planned L
    L1 = S.plan_bins(N, K, 0.9)
    v, i = S.approx_max_k(t[:50], K, recall_target=0.9, aggregate_to_topk=False)
    assert v.shape == (50, min(L1, N))
    L2 = min(S.plan_bins(10 * N, K, 0.99), N)
    v, i = S.approx_max_k(t[:50], K, recall_target=0.99, planning_size=10 * N,
                          aggregate_to_topk=False)
    assert v.shape == (50, L2)
    ov, oi = oracle.approx_max_k(X[:50].astype(np.float64), K, L2, aggregate_to_topk=False)
    assert np.array_equal(i.cpu().numpy(), oi)


@pytest.mark.parametrize("bins", ["mod", "contiguous"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("N", [4096, 5000, 70000])
def test_approx_max_k_16_byte_loads_match_oracle(bins, dtype, N):
    """L (j mod L bins) and N multiples of the columns one 16-byte load holds
    (4 FP32, 8 BF16): the vectorised kernels, bit-exact against the oracle
    including ties and zeros of both signs, rows, grid rows and column runs
    split over many CTAs (70000 columns span several CTAs of a row)."""
    ensure_built()
    M, K = 37, 10
    X = scores(M, N, 43)
    t = torch.from_numpy(X).cuda()
    if dtype == "bf16":
        t = t.to(torch.bfloat16)
    Xo = t.float().cpu().numpy().astype(np.float64)
    for L in (8, 64, 1000, N):
        for is_min in (False, True):
            for agg in (False, True):
                k = min(K, L)
                v, i = S.approx_max_k(t, k, L=L, bins=bins, is_min=is_min, aggregate_to_topk=agg)
                ov, oi = oracle.approx_max_k(Xo, k, L, bins=bins, is_min=is_min,
                                             aggregate_to_topk=agg)
                v, i = v.cpu().numpy(), i.cpu().numpy()
                assert np.array_equal(i, oi), (L, is_min, agg)
                assert np.array_equal(v.astype(np.float64), ov), (L, is_min, agg)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("M,N,L", [(3, 1, 1), (2, 9, 8), (5, 4096, 8), (7, 40_003, 1), (3, 40_000, 176),
                                   (2, 100_003, 1931), (4, 65_536, 2048), (2, 70_000, 2064),
                                   (1, 300_007, 255), (1, 300_000, 40)])
def test_approx_max_k_grid_rows(M, N, L, dtype):
    """Bin winners where the kernel's threads share a grid row's vectors and
    several grid rows: few and many bins, 16-byte loads and single ones, a
    ragged last grid row, more vectors than one block's threads."""
    ensure_built()
    X = scores(M, N, 43 + L)
    t = torch.from_numpy(X).cuda()
    if dtype == "bf16":
        t = t.to(torch.bfloat16)
    Xo = t.float().cpu().numpy().astype(np.float64)
    for is_min in (False, True):
        v, i = S.approx_max_k(t, 1, L=L, is_min=is_min, aggregate_to_topk=False)
        ov, oi = oracle.approx_max_k(Xo, 1, L, is_min=is_min, aggregate_to_topk=False)
        assert np.array_equal(i.cpu().numpy(), oi)
        assert np.array_equal(v.cpu().numpy().astype(np.float64), ov)


@pytest.mark.parametrize("bins", ["mod", "contiguous"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_approx_max_k_nan_comes_first(bins, dtype):
    """One rule for NaN (before every other score, the smaller column among
    several), the same with 16-byte loads and with single ones (the matrix
    starting one element later): NaN in the first, a middle and the last grid
    row of a bin, twice in a bin, beside infinities, and bins of -inf alone."""
    ensure_built()
    M, N = 4, 8192
    g = np.random.Generator(np.random.PCG64(51))
    X = g.standard_normal((M, N)).astype(np.float32)
    X[0, [3, 4099, 8191]] = np.nan
    X[1, [100, 101, 4000, 4001, 5000]] = [np.nan, np.inf, np.inf, np.nan, -np.inf]
    X[2, :] = -np.inf
    X[2, [7, 4103]] = np.nan
    X[3, :] = np.inf
    X[3, 8000] = np.nan
    flat = torch.empty(M * N + 1, device="cuda")
    flat[1:] = torch.from_numpy(X).cuda().reshape(-1)
    if dtype == "bf16":
        flat = flat.to(torch.bfloat16)
    shifted = flat[1:].view(M, N)
    Xo = shifted.float().cpu().numpy().astype(np.float64)
    for is_min in (False, True):
        rank = np.clip(-Xo if is_min else Xo, -1e200, 1e200)
        rank[np.isnan(Xo)] = 1e300
        for L in (8, 64, 176, 4096, N):
            j = np.arange(N)
            q, r = N // L, N % L
            b = j % L if bins == "mod" else np.where(j < r * (q + 1), j // (q + 1),
                                                     r + (j - r * (q + 1)) // q)
            first = np.array([[np.flatnonzero(b == t)[np.argmax(rank[i, b == t])]
                               for t in range(L)] for i in range(M)])
            for t in (shifted, shifted.clone()):
                v, i = S.approx_max_k(t, 1, L=L, bins=bins, is_min=is_min, aggregate_to_topk=False)
                np.testing.assert_array_equal(i.cpu().numpy(), first)
                np.testing.assert_array_equal(v.cpu().numpy().astype(np.float64),
                                              np.take_along_axis(Xo, first, 1))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("M,N,L", [(1, 300_000, 8), (1, 262_144, 2064), (3, 65_536, 128),
                                   (65, 4096, 128), (66, 4099, 128), (1000, 1024, 8), (300, 513, 40),
                                   (67, 64, 8), (70_001, 24, 8), (5, 1000, 1)])
def test_approx_max_k_work_split(M, N, L, dtype):
    """How rows, grid rows and bins are shared out over threads and CTAs: many
    chunks of one row, several rows to a CTA (the last CTA part empty), more
    rows than one launch takes; integers, so ties keep the smaller column."""
    ensure_built()
    g = torch.Generator(device="cuda")
    g.manual_seed(N + L)
    t = torch.randint(-9, 10, (M, N), generator=g, device="cuda").float()
    if dtype == "bf16":
        t = t.to(torch.bfloat16)
    T = (N + L - 1) // L
    s = torch.full((M, T * L), -float("inf"), device="cuda")
    s[:, :N] = t.float()
    s = s.view(M, T, L)
    best = s.amax(1)
    first = (s == best[:, None, :]).float().argmax(1)
    v, i = S.approx_max_k(t, 1, L=L, aggregate_to_topk=False)
    assert torch.equal(v, best)
    assert torch.equal(i.long(), first * L + torch.arange(L, device="cuda")[None, :])


def us(f):
    for _ in range(3):
        f()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t = []
    for _ in range(11):
        a.record()
        for _ in range(8):       # (of one call the host takes as long)
            f()
        b.record()
        b.synchronize()
        t.append(a.elapsed_time(b))
    return min(t)


def test_approx_max_k_of_many_short_rows():
    """20,000 rows of 1024 scores take about as long as 5000 rows of 4096 (with
    all of a CTA's threads over one row's 128 grid rows, twice as long)."""
    ensure_built()
    t = torch.zeros((5000, 4096), device="cuda")
    long_rows = us(lambda: S.approx_max_k(t, 1, L=8, aggregate_to_topk=False))
    t = t.view(20_000, 1024)
    short_rows = us(lambda: S.approx_max_k(t, 1, L=8, aggregate_to_topk=False))
    assert short_rows < 1.5 * long_rows
