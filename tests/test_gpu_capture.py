"""k-NN calls recorded into a CUDA graph while the buffer has no current tree:
the capture leaves the forest as it was (a tree that it built would exist only
once the graph has run), so that calls before the first replay, the replays
and calls after them all give the exact rows."""
import numpy as np
import pytest
import torch

from oracle.threads import bruteforce_knn_threads
from paper_2112_06188_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_06188_gb300 import build_lib
    build_lib.build()


@pytest.mark.parametrize("calls_before", [0, 1, 2])
@pytest.mark.parametrize("dim,m,k,split", [(2, 300, 5, "object"), (3, 20_000, 8, "spatial"), (5, 100, 3, "object")])
def test_capture_with_a_changed_buffer(calls_before, dim, m, k, split, monkeypatch):
    from paper_2112_06188_gb300.forest import Forest
    monkeypatch.setenv("BDL_DEBUG_CHECK", "0")   # (its wait after every call cannot be captured)
    warm = Forest(dim, split=split)         # loads the kernels (a capture cannot)
    warm.insert(torch.from_numpy(inputs.uniform_points(5_000, dim, 1)).cuda())
    f, live = Forest(dim, split=split), inputs.LiveSet(dim)
    q = inputs.uniform_points(m, dim, 9)
    dq = torch.from_numpy(q).cuda()
    warm.knn(dq, k)
    new = lambda: (torch.full((m, k), -7, dtype=torch.int32, device="cuda"), torch.full((m, k), -7, dtype=torch.int64, device="cuda"))

    def check(got):
        torch.cuda.synchronize()
        pts, ids = live.live_points()
        bi, bd = bruteforce_knn_threads(pts, ids, q, k)
        assert np.array_equal(got[1].cpu().numpy(), bd) and np.array_equal(got[0].cpu().numpy(), bi)

    for step, n in enumerate((5_700, 40)):
        p = inputs.uniform_points(n, dim, 20 + step)
        f.insert(torch.from_numpy(p).cuda())
        live.insert(p)
        for _ in range(calls_before):
            check(f.knn(dq, k, out=new()))
        out = new()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            f.knn(dq, k, out=out)
        check(f.knn(dq, k, out=new()))      # before the first replay
        for _ in range(2):
            out[0].fill_(-7)
            out[1].fill_(-7)
            g.replay()
            check(out)
        check(f.knn(dq, k, out=new()))
        del g
    assert f.poll_error() == 0
    f.close()
