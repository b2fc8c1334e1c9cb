"""Searches from several host threads at once: the library's calls release the
interpreter's lock, so their host code runs side by side."""
import threading

import pytest
import torch

from paper_2206_14286_gb300 import search as S
from tests.gpu_util import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,D,Ms", [("bf16", 64, (1, 120)), ("bf16", 256, (8, 128)),
                                        ("f32", 32, (70, 600)), ("e4m3", 64, (5, 60))])
def test_threads_with_different_batch_sizes(dtype, D, Ms):
    """Threads that search one database with different numbers of queries launch
    the same kernels with different shared memory; every call goes through, with
    the results of the same call alone."""
    ensure_built()
    g = torch.Generator(device="cuda")
    g.manual_seed(D)
    d = S.Database(torch.randn((3000, D), generator=g, device="cuda"), metric="ip", dtype=dtype)
    qs = [torch.randn((M, D), generator=g, device="cuda") for M in Ms]
    want = [tuple(t.clone() for t in d.search(q, 8, L=64)) for q in qs]
    torch.cuda.synchronize()
    failed = []
    start = threading.Barrier(2 * len(qs))

    def work(k, slot):
        try:
            st = torch.cuda.Stream()
            out = (torch.empty_like(want[k][0]), torch.empty_like(want[k][1]))
            start.wait()
            for _ in range(3000):
                d.search(qs[k], 8, L=64, stream=st, out=out, slot=slot)
            st.synchronize()
            if not (torch.equal(out[0], want[k][0]) and torch.equal(out[1], want[k][1])):
                failed.append("other results for %d queries" % Ms[k])
        except Exception as e:                              # noqa: BLE001
            failed.append("%d queries: %s" % (Ms[k], e))

    threads = [threading.Thread(target=work, args=(k, "t%d%d" % (k, r)))
               for k in range(len(qs)) for r in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
