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
