"""The plans that Database keeps for the sizes that come again (host side; the
library's sizes need no GPU)."""
import numpy as np
import pytest
import torch

from paper_2206_14286_gb300 import _lib
from paper_2206_14286_gb300 import build as B
from paper_2206_14286_gb300 import search as S
from paper_2206_14286_gb300._lib import DTYPE, METRIC


def database(N=100_000, D=64):
    B.build()
    d = object.__new__(S.Database)
    d.N, d.D, d.metric, d.dtype, d._plans = N, D, "l2", "bf16", {}
    return d


@pytest.mark.parametrize("make", [lambda v: torch.tensor(v), lambda v: np.array(v)[()]])
def test_plans_are_kept_by_value(make):
    """An argument that is changed in place gets the plan of its new value."""
    d = database()
    want = {K: database()._search_plan(8, K, None, 0.95, 2, "mod") for K in (5, 50)}
    assert want[5] != want[50]
    K = make(5)
    assert d._search_plan(8, K, None, 0.95, 2, "mod") == want[5]
    if isinstance(K, torch.Tensor):
        K.fill_(50)
    else:
        K = make(50)
    assert d._search_plan(8, K, None, 0.95, 2, "mod") == want[50]
    assert d._search_plan(8, 5, None, 0.95, 2, "mod") == want[5]


def test_plans_are_bounded():
    d = database()
    for M in range(1, 600):
        d._search_plan(M, 10, 1000, 0.95, 2, "mod")
        assert len(d._plans) <= 256


def test_exact_workspace_of_large_k_holds_one_running_set():
    """Beyond 1024 results the running set is updated in place: 500 more of them
    for 128 queries are 500 x 128 keys."""
    B.build()
    ws = [_lib.get().knn_search_exact_workspace(100_000, 64, DTYPE["f32"], METRIC["l2"], 128, K)
          for K in (1500, 2000)]
    assert ws[1] - ws[0] == 500 * 128 * 8
