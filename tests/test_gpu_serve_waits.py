"""The request server holds small k-NN requests of a burst back for up to 300
us so that they share a launch, but never one that a caller waits for: a client
that asks, waits and asks again gets each answer at once, also while finished
tickets lie uncollected and when it waits by draining."""
import time

import numpy as np
import pytest
import torch

from paper_2112_06188_gb300 import inputs

pytestmark = pytest.mark.gpu

N = 30
HELD_MS = 0.3      # what a request may be held back


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_06188_gb300 import build_lib
    build_lib.build()


@pytest.fixture(scope="module")
def server():
    from paper_2112_06188_gb300.forest import Forest
    from paper_2112_06188_gb300.serve import Server
    f = Forest(2)
    f.insert(torch.from_numpy(inputs.uniform_points(20_000, 2, 3)).cuda())
    torch.cuda.synchronize()
    s = Server(f)
    yield s
    s.close()
    f.close()


def request(m=8, k=4):
    q = torch.from_numpy(inputs.uniform_points(m, 2, 5)).pin_memory()
    return q, k, (torch.empty((m, k), dtype=torch.int32).pin_memory(), torch.empty((m, k), dtype=torch.int64).pin_memory())


@pytest.mark.parametrize("uncollected", [0, 1, 20])
@pytest.mark.parametrize("by_drain", [False, True])
def test_asking_and_waiting_in_turn(server, uncollected, by_drain):
    s = server
    q, k, out = request()
    left = [s.knn(*request()[:2]) for _ in range(uncollected)]
    s.drain()
    best = 1e9
    for _ in range(8):
        tickets = []
        t0 = time.perf_counter()
        for _ in range(N):
            t = s.knn(q, k, out=out)
            if by_drain:
                s.drain()
                tickets.append(t)
            else:
                s.wait(t)
        best = min(best, (time.perf_counter() - t0) * 1e3)
        left += tickets
    for t in left:
        s.wait(t)
    # every group held back until 300 us after the last one: N - 1 such gaps at least
    assert best < (N - 1) * HELD_MS


def test_small_budget_does_not_hold_back(server):
    """Staging memory for one request only: a second one cannot join the first."""
    from paper_2112_06188_gb300.serve import Server
    q, k, _ = request()
    s = Server(server.forest, staging_budget_bytes=q.numel() * 4 + 8 * k * 12)
    best = 1e9
    for _ in range(8):
        outs = [request()[2] for _ in range(N)]
        t0 = time.perf_counter()
        tickets = [s.knn(q, k, out=o) for o in outs]
        for t in tickets:
            s.wait(t)
        best = min(best, (time.perf_counter() - t0) * 1e3)
    assert s.groups() == 8 * N
    s.close()
    assert best < (N - 1) * HELD_MS
    want = outs[0]
    for o in outs[1:]:
        assert np.array_equal(o[0].numpy(), want[0].numpy()) and np.array_equal(o[1].numpy(), want[1].numpy())
