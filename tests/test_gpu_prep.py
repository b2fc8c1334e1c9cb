"""Row preparation bit for bit against the FP64 definition (the oracle's), at
the edges of its row-length variants and where the paired-FP32 arithmetic has
to hand a row to FP64: zero and tiny rows, huge rows, signed zeros, infinities
and NaN, unaligned rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_2206_14286_gb300 import search as S
from tests.gpu_util import ensure_built

pytestmark = pytest.mark.gpu


def rows_of(rows, D, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    X = g.standard_normal((rows, D)).astype(np.float32)
    X *= np.exp(g.uniform(-3, 3, (rows, 1))).astype(np.float32)
    X[::5, ::3] = -0.0
    X[1] = 0.0
    X[2] = -0.0
    X[3] *= np.float32(2.0 ** -70)
    X[4] *= np.float32(2.0 ** 60)
    X[5, 0] = np.float32(2.0 ** -140)
    X[6] = np.float32(1.0)               # |x|^2 = D: exact squares and ties
    X[7] = 0.0
    X[7, D - 1] = np.float32(3.0)
    return X


@pytest.mark.parametrize("D", [1, 3, 16, 63, 64, 65, 96, 97, 128, 129, 255, 256, 257, 512, 513,
                               1024, 1025, 1500, 4096])
def test_prepare_bits_at_every_row_length(D):
    ensure_built()
    rows = 1501
    X = rows_of(rows, D, 100 + D)
    # rows starting on a 4-byte boundary that is not a 16-byte one, too
    flat = torch.empty(rows * D + 1, device="cuda")
    flat[1:] = torch.from_numpy(X).cuda().reshape(-1)
    unit = oracle.normalize_rows(X)
    for x in (torch.from_numpy(X).cuda(), flat[1:].view(rows, D)):
        for dtype in ("f32", "bf16", "e4m3"):
            d = S.Database(x, metric="cos", dtype=dtype)
            got = d.f32.cpu().numpy()
            np.testing.assert_array_equal(got.view(np.uint32), unit.view(np.uint32))
            if dtype == "e4m3":
                ref, sc = oracle.e4m3_rows(unit)
                np.testing.assert_array_equal(d.scale.cpu().numpy(), sc)
                lp = d.lp.view(torch.float8_e4m3fn).reshape(rows, d.pitch).float().cpu().numpy()
                val = lp[:, :D].astype(np.float64) * sc[:, None].astype(np.float64)
            else:
                t = torch.bfloat16 if dtype == "bf16" else torch.float32
                lp = d.lp.view(t).reshape(rows, d.pitch).float().cpu().numpy()
                val = lp[:, :D].astype(np.float64)
                ref = oracle.bf16_round(unit) if dtype == "bf16" else unit.astype(np.float64)
            np.testing.assert_array_equal(val, ref)
            assert (lp[:, D:] == 0).all()
        # L2 half norms: half the FP64 sum of the squares of the stored values
        # in FP32 (an E4M3 code times its scale rounds once), rounded once
        # (rows 3 and 4 leave FP32's range: 0 and inf)
        for dtype, ref in (("f32", X.astype(np.float64)), ("bf16", oracle.bf16_round(X)),
                           ("e4m3", oracle.e4m3_rows(X)[0].astype(np.float32).astype(float))):
            d = S.Database(x, metric="l2", dtype=dtype)
            with np.errstate(over="ignore"):
                h = (0.5 * (ref * ref).sum(1)).astype(np.float32)
            np.testing.assert_array_equal(d.hnorm.cpu().numpy(), h)


@pytest.mark.parametrize("D", [40, 96, 300, 1100])
def test_prepare_infinities_and_nan(D):
    """A row with an infinity or a NaN comes out as FP64 leaves it (its unit
    row has NaN where inf * 0 or NaN entered, 0 elsewhere for an infinity),
    its padding stays zero, and its neighbours in the warp are untouched."""
    ensure_built()
    rows = 64
    X = rows_of(rows, D, 7 + D)
    X[9, D // 2] = np.inf
    X[17, 0] = np.nan
    unit = oracle.normalize_rows(X)
    for dtype in ("f32", "bf16", "e4m3"):
        d = S.Database(torch.from_numpy(X).cuda(), metric="cos", dtype=dtype)
        got = d.f32.cpu().numpy()
        for r in range(rows):
            if r == 9:
                assert np.isnan(got[r, D // 2]) and (np.delete(got[r], D // 2) == 0).all()
            elif r == 17:
                assert np.isnan(got[r]).all()
            else:
                np.testing.assert_array_equal(got[r].view(np.uint32), unit[r].view(np.uint32))
        if dtype != "e4m3":
            t = torch.bfloat16 if dtype == "bf16" else torch.float32
            lp = d.lp.view(t).reshape(rows, d.pitch).float().cpu().numpy()
            assert (lp[:, D:] == 0).all()


# 1024-element rows of 1022 times 2^50, then w 2^26, then v 2^7, (w, v) below:
# the inverse norm's square is so small that FP32 holds it in a subnormal's few
# bits, and v times the inverse norm lies within 2^-44 of a rounding midpoint,
# so paired FP32 that took the inverse for good here rounds v to the other side
# (found by exact evaluation of its steps). The hardware's reciprocal square
# root may be off by a few units in the last place; rows for each.
NEAR_2_50 = [
    # off by -2 units in the last place
    (0xee2d69, 0x85bacf), (0xee2d69, 0xa39114), (0xeb7ac2, 0x9bd93c), (0xeb7ac2, 0xbaab52), (0xd3772e, 0x9a354b),
    (0xd3772e, 0xde10e1), (0xd411cd, 0x90af9d), (0xd411cd, 0x9eaed1), (0xbe7dea, 0x842046), (0xbe7dea, 0x90b5a2),
    # off by -1 units in the last place
    (0xf93989, 0xa4beec), (0xf93989, 0xc862f5), (0xcf3c70, 0xb91e72), (0x91b8d6, 0xd28106), (0xcae018, 0xa8d3c8),
    (0xcae018, 0xc9c0ca), (0xec993f, 0xa87206), (0xb20fe8, 0xdb1b11), (0xb20fe8, 0xf5c456), (0xcdffbc, 0xfd28ee),
    # off by 0 units in the last place
    (0xb4f2af, 0xcb9648), (0xc33596, 0xd6b008), (0xa576bb, 0x9de3c2), (0x89a947, 0xdb5854), (0x89a947, 0xdc1323),
    (0x96160a, 0xa212cf), (0x96160a, 0xe97ea6), (0xfac950, 0xb4242a), (0x89a915, 0xfe3051), (0xc33574, 0x91f5c1),
    # off by 1 units in the last place
    (0xf8472b, 0xfa6668), (0x80272e, 0x8474ab), (0x99866a, 0xeb1e4b), (0xa58ae2, 0xa277c8), (0xa58ae2, 0xb61a0e),
    (0xdec760, 0x8531d7), (0xdec760, 0xfaf361), (0xf94e31, 0xf2c1d0), (0xfee1f8, 0xd30530), (0xfee1f8, 0xe6072d),
    # off by 2 units in the last place
    (0xe7ce45, 0x876d2e), (0xe7ce45, 0x8d091f), (0xf746ac, 0xfe53cd), (0x8e5db9, 0x937372), (0x8e5db9, 0xe15f1c),
    (0xca616d, 0x82b7a9), (0xca616d, 0xa1356d), (0x8f42a5, 0x8a9d57), (0x8f42a5, 0xcdbe42), (0x955ead, 0xceda8d),
]


def test_prepare_bits_of_huge_norms():
    ensure_built()
    X = np.full((len(NEAR_2_50), 1024), 2.0 ** 50, np.float32)
    X[:, 1022] = [w * 2.0 ** 26 for w, _ in NEAR_2_50]
    X[:, 1023] = [v * 2.0 ** 7 for _, v in NEAR_2_50]
    unit = oracle.normalize_rows(X)
    for dtype in ("f32", "bf16", "e4m3"):
        d = S.Database(torch.from_numpy(X).cuda(), metric="cos", dtype=dtype)
        np.testing.assert_array_equal(d.f32.cpu().numpy().view(np.uint32), unit.view(np.uint32))


@pytest.mark.parametrize("D", [64, 257, 1024, 1500, 4096])
def test_prepare_bits_at_the_ends_of_the_paired_range(D):
    """Rows whose largest element is at, just inside and just outside each end
    of the range that paired FP32 handles (2^-40 and 2^40)."""
    ensure_built()
    g = np.random.Generator(np.random.PCG64(D))
    tops = [np.float32(2.0 ** e) for e in (-41, -40, -39, 39, 40, 41, 50)]
    tops += [np.nextafter(t, np.float32(s)) for t in tops for s in (0.0, np.inf)]
    X = (g.uniform(0.5, 1.0, (16 * len(tops), D)) * g.choice([-1.0, 1.0], (16 * len(tops), D)))
    X = (X * np.repeat(np.array(tops, np.float64), 16)[:, None]).astype(np.float32)
    X[:, 0] = np.repeat(np.array(tops, np.float32), 16)
    unit = oracle.normalize_rows(X)
    d = S.Database(torch.from_numpy(X).cuda(), metric="cos", dtype="f32")
    np.testing.assert_array_equal(d.f32.cpu().numpy().view(np.uint32), unit.view(np.uint32))
    d = S.Database(torch.from_numpy(X).cuda(), metric="l2", dtype="f32")
    X64 = X.astype(np.float64)
    np.testing.assert_array_equal(d.hnorm.cpu().numpy(), (0.5 * (X64 * X64).sum(1)).astype(np.float32))


@pytest.mark.parametrize("D", [64, 257, 1024, 1500, 4096])
def test_half_norms_of_small_rows(D):
    """L2 half norms of rows of zeros (of either sign, with a NaN or not) and
    around the lower end of the range that paired FP32 handles (2^-50)."""
    ensure_built()
    g = np.random.Generator(np.random.PCG64(D + 1))
    tops = [2.0 ** e for e in (-70, -52, -51, -50, -49, -45)]
    tops += [np.nextafter(np.float32(2.0 ** -50), np.float32(0.0))]
    X = g.uniform(0.25, 1.0, (32 * len(tops), D)) * np.repeat(tops, 32)[:, None]
    X[:, ::3] *= 2.0 ** -12                     # squares that lose bits
    X[:, 0] = np.repeat(tops, 32)
    X = X.astype(np.float32)
    X[5] = 0.0
    X[6] = -0.0
    X[7] = 0.0
    X[7, D // 2] = np.nan
    X[8] = 0.0
    X[8, D - 1] = np.float32(2.0 ** -140)
    d = S.Database(torch.from_numpy(X).cuda(), metric="l2", dtype="f32")
    X64 = X.astype(np.float64)
    h = (0.5 * (X64 * X64).sum(1)).astype(np.float32)
    np.testing.assert_array_equal(d.hnorm.cpu().numpy(), h)


def test_rows_of_zeros_cost_no_more_than_others():
    """(in FP64 beside the paired FP32, 3 times as much)"""
    ensure_built()

    def ms(x):
        for _ in range(3):
            S.Database(x, metric="l2", dtype="f32")
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t = []
        for _ in range(9):
            a.record()
            for _ in range(8):
                S.Database(x, metric="l2", dtype="f32")
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        return min(t)

    x = torch.randn((50_000, 257), device="cuda")
    assert ms(torch.zeros_like(x)) < 1.5 * ms(x)
