"""The tensor-core PartialReduce at the edges of its work split: one or two
query halves per tile (M around multiples of 8 and 128), the two bin grids (N
a multiple of L or not, T + 1 crossing a group of 16 grid rows), virtual bins
(few bins folded over L), every K-loop mode, both bin maps -- against scores of
the same stored values in 64 bits."""
import pytest
import torch

from paper_2206_14286_gb300 import search as S
from tests.gpu_util import ensure_built

pytestmark = pytest.mark.gpu


def scores64(d, q, dtype):
    """FP64 scores of the values the contraction saw, and the natural scale."""
    D = d.D
    if dtype == "bf16":
        xs = d.lp.view(torch.bfloat16).view(d.N, d.pitch)[:, :D].double()
        qs = q.to(torch.bfloat16).double()
    else:
        s = d.scale.double()[:, None]
        xs = d.lp.view(torch.float8_e4m3fn).view(d.N, d.pitch)[:, :D].float().double() * s
        # the kernel leaves the per-query scale out of the value
        # (a true division: by a Python number torch multiplies by its inverse)
        qsc = q.abs().amax(1, keepdim=True) / torch.full((q.shape[0], 1), 448.0, device="cuda")
        qs = (q / qsc).to(torch.float8_e4m3fn).double()
    s = qs @ xs.t()
    if d.metric == "l2":
        s = s - 0.5 * (xs * xs).sum(1)[None, :]
    scale = qs.norm(dim=1)[:, None] * xs.norm(dim=1).max()
    if d.metric == "l2":
        scale = scale + 0.5 * (xs * xs).sum(1).max()
    return s, scale


def bin_of(N, L, bins):
    j = torch.arange(N, device="cuda")
    if bins == "mod":
        return j % L
    q, r = N // L, N % L
    big = r * (q + 1)
    return torch.where(j < big, j // (q + 1), r + (j - big) // max(q, 1))


@pytest.mark.parametrize("dtype,metric", [("bf16", "l2"), ("bf16", "ip"), ("e4m3t", "ip")])
@pytest.mark.parametrize("M", [1, 7, 8, 9, 33, 127, 128, 129, 256, 257, 333, 513])
@pytest.mark.parametrize("N,L,D", [
    (4096, 16, 128),      # no ragged row, T a multiple of 16
    (4097, 16, 128),      # a ragged row that starts a group of 16 grid rows
    (40_011, 20, 100),    # virtual bins, odd row length
    (30_000, 3, 16),      # very few bins
    (12_345, 1, 64),      # one bin
    (9_999, 1931, 40),    # fewer than 16 grid rows
    (5_003, 605, 256),    # K loop, resident queries
    (3_001, 77, 768),     # K loop, streamed queries (resident when few)
])
def test_partial_reduce_work_split(dtype, metric, M, N, L, D):
    ensure_built()
    g = torch.Generator(device="cuda")
    g.manual_seed(N + 31 * M + D)
    x = torch.randn((N, D), generator=g, device="cuda")
    q = torch.randn((M, D), generator=g, device="cuda")
    d = S.Database(x, metric=metric, dtype=dtype)
    s, scale = scores64(d, q, dtype)
    # FP32 accumulation of D exact products (tensor-core rounding toward zero:
    # 2^-23 of the running magnitude a step) and the three-part BF16 half norm
    tol = (D + 16) * 2.0 ** -23 * scale + (2.0 ** -20 * scale if metric == "l2" else 0.0)
    for bins in ("mod", "contiguous"):
        V, A = d.partial_reduce(q, L, bins=bins)
        S.sync_status()
        b = bin_of(N, L, bins)
        best = torch.full((M, L), -float("inf"), dtype=torch.float64, device="cuda")
        best.scatter_reduce_(1, b[None, :].expand(M, N), s, "amax")
        A = A.long()
        assert ((A >= 0) & (A < N)).all()
        assert (b[A] == torch.arange(L, device="cuda")[None, :]).all()
        own = s.gather(1, A)
        assert ((V.double() - own).abs() <= tol).all()     # the value is its row's score
        assert (best - own <= 2 * tol).all()               # and the bin's best


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


def test_fp32_tiles_of_a_cta_per_sm_spread_over_the_sms():
    """144 CTAs of one tile each take no longer than 48 of them, give or take
    their share of the memory system (two to an SM they took 1.6 times as long)."""
    ensure_built()
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    x = torch.randn((3000, 4096), generator=g, device="cuda")
    q = torch.randn((333, 4096), generator=g, device="cuda")
    d = S.Database(x, metric="ip", dtype="f32")
    assert us(lambda: d.partial_reduce(q, 1024)) < 1.3 * us(lambda: d.partial_reduce(q[:128], 1024))


@pytest.mark.parametrize("M,N,L", [(333, 3000, 605), (1000, 3000, 1024), (65, 9000, 1024),
                                   (70, 20_000, 2000), (7, 100, 3)])
def test_fp32_partial_reduce_launches(M, N, L):
    """The FP32 kernel's launches (an SM to each CTA, in order, early), on
    integers: exact scores and the smaller row on ties."""
    ensure_built()
    g = torch.Generator(device="cuda")
    g.manual_seed(M)
    x = torch.randint(-2, 3, (N, 20), generator=g, device="cuda").float()
    q = torch.randint(-2, 3, (M, 20), generator=g, device="cuda").float()
    V, A = S.Database(x, metric="ip", dtype="f32").partial_reduce(q, L)
    # the bins' columns side by side, -inf past the last row; the first maximum
    T = (N + L - 1) // L
    s = torch.full((M, T * L), -float("inf"), device="cuda")
    s[:, :N] = q @ x.t()
    s = s.view(M, T, L)
    best = s.amax(1)
    first = (s == best[:, None, :]).float().argmax(1)
    assert torch.equal(V, best)
    assert torch.equal(A.long(), first * L + torch.arange(L, device="cuda")[None, :])


def test_few_bins_do_not_queue_for_their_keys():
    """Three bins of a small database take about as long as twenty (with five
    virtual bins each, all CTAs merging into the same few keys, 2.3 times)."""
    ensure_built()
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    x = torch.randn((60_000, 64), generator=g, device="cuda")
    q = torch.randn((64, 64), generator=g, device="cuda")
    d = S.Database(x, metric="ip", dtype="bf16")
    assert us(lambda: d.partial_reduce(q, 3)) < 1.6 * us(lambda: d.partial_reduce(q, 20))


def schedule(nqt, steps, sms):
    """(tiles per CTA, steps per CTA) of the tensor-core kernel's host schedule."""
    first = (nqt + sms - 1) // sms
    best = None
    for kq in range(first, min(nqt, first + 16) + 1):
        groups = (nqt + kq - 1) // kq
        if groups > sms:
            continue
        parts = min(sms // groups, steps)
        spp = (steps + parts - 1) // parts
        if best is None or kq * (spp + 1) < best[0]:
            best = (kq * (spp + 1), kq, spp)
    return best[1:]


@pytest.mark.parametrize("bins", ["mod", "contiguous"])
def test_l2_half_norms_of_several_tiles_per_cta(bins):
    """A CTA that takes several query tiles in turn over its rows starts the
    rows' half norms again with each, while the next tile's are already on
    their way, and (contiguous bins) the first bin of its rows."""
    ensure_built()
    D, M = 64, 3339
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    odd = 0
    for N, L in ((100_000, 605), (91_000, 333)):
        T, r = N // L, N % L
        up = lambda a, b: (a + b - 1) // b
        steps = (up(r, 16) * up(T + 1, 16) + up(L - r, 16) * up(T, 16) if bins == "mod"
                 else up(N, 256))
        two, one = schedule(up(M, 256), steps, sms), schedule(up(M, 128), steps, sms)
        factor = 1.1 if bins == "mod" else 1.5
        kq, spp = one if factor * one[0] * (one[1] + 1) < 2.0 * two[0] * (two[1] + 1) else two
        assert kq >= 2
        odd += spp % 2
        g = torch.Generator(device="cuda")
        g.manual_seed(L)
        x = torch.randint(-2, 3, (N, D), generator=g, device="cuda").float()
        q = torch.randint(-2, 3, (M, D), generator=g, device="cuda").float()
        d = S.Database(x, metric="l2", dtype="bf16")
        V, A = d.partial_reduce(q, L, bins=bins)
        S.sync_status()
        s = q @ x.t() - 0.5 * (x * x).sum(1)[None, :]
        best, first = bin_winners(s, L, bins)
        assert torch.equal(V, best)
        assert torch.equal(A.long(), first)
        del s, best, first
    assert odd          # an odd number of steps per tile, too


def bin_winners(s, L, bins):
    """(best score, first row that has it) of each bin, M x L."""
    M, N = s.shape
    j = torch.arange(N, device=s.device)
    b = bin_of(N, L, bins)[None, :].expand(M, N)
    best = torch.full((M, L), -float("inf"), device=s.device).scatter_reduce(1, b, s, "amax")
    at = torch.where(s == best.gather(1, b), j[None, :], N)
    first = torch.full((M, L), N, device=s.device).scatter_reduce(1, b, at, "amin")
    return best, first


@pytest.mark.parametrize("dtype,metric", [("bf16", "ip"), ("bf16", "l2"), ("e4m3t", "ip")])
@pytest.mark.parametrize("M", [1, 128, 129, 333])
@pytest.mark.parametrize("N,L", [(40_011, 3), (40_011, 20), (40_011, 605), (4097, 16), (300, 77)])
def test_partial_reduce_ties_keep_the_smaller_row(dtype, metric, M, N, L):
    """Integers, whose scores are exact and mostly tie: through virtual bins,
    both grids, accumulators that take alternate steps and the search for a
    run's position."""
    ensure_built()
    g = torch.Generator(device="cuda")
    g.manual_seed(N + L + M)
    x = torch.randint(-2, 3, (N, 24), generator=g, device="cuda").float()
    q = torch.randint(-2, 3, (M, 24), generator=g, device="cuda").float()
    if dtype == "e4m3t":          # scales 1: the codes are the values
        x[:, 0], q[:, 0] = 448.0, 448.0
    s = q @ x.t()
    if metric == "l2":
        s = s - 0.5 * (x * x).sum(1)[None, :]
    d = S.Database(x, metric=metric, dtype=dtype)
    for bins in ("mod", "contiguous"):
        V, A = d.partial_reduce(q, L, bins=bins)
        best, first = bin_winners(s, L, bins)
        assert torch.equal(V, best)
        assert torch.equal(A.long(), first)
