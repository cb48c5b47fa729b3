"""When a k-NN call builds the buffer's tree: the first call on a forest and
after a change does, unless the caller asked exactly once between the last
changes (then a small first call scans and a second one builds); calls without
allocation, batches and plans count.  Rows against brute force throughout."""
import ctypes

import numpy as np
import pytest
import torch

from oracle.threads import bruteforce_knn_threads
from paper_2112_06188_gb300 import inputs

pytestmark = pytest.mark.gpu
K = 6


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_06188_gb300 import build_lib
    build_lib.build()


class Case:
    """A forest with a part-filled buffer; `ask` and the others return whether the call built a tree."""

    def __init__(self, dim, m=40, X=1024, nbuf=700, split="object"):
        from paper_2112_06188_gb300.forest import Forest
        self.f, self.live = Forest(dim, buffer_size=X, split=split), inputs.LiveSet(dim)
        self.kernel = "k_subtree" if split == "object" else "k_sp_levels"
        self.dim, self.seed = dim, 10 * dim
        self.q = inputs.uniform_points(m, dim, 5)
        self.dq = torch.from_numpy(self.q).cuda()
        self.change(3 * X + nbuf)

    def change(self, n=3):
        self.seed += 1
        p = inputs.uniform_points(n, self.dim, self.seed)
        self.f.insert(torch.from_numpy(p).cuda())
        self.live.insert(p)

    def run(self, call):
        from paper_2112_06188_gb300 import capi
        torch.cuda.synchronize()
        capi.bdl_profile(1)
        rows = call()
        torch.cuda.synchronize()
        built = self.kernel in capi.bdl_profile_read()
        capi.bdl_profile(0)
        pts, ids = self.live.live_points()
        bi, bd = bruteforce_knn_threads(pts, ids, self.q, K)
        for gi, gd in rows:
            assert np.array_equal(gi.cpu().numpy(), bi) and np.array_equal(gd.cpu().numpy(), bd)
        return built

    def ask(self):
        return self.run(lambda: [self.f.knn(self.dq, K)])

    def ask_twice_in_a_batch(self):
        from paper_2112_06188_gb300.forest import knn_batch
        return self.run(lambda: knn_batch([self.f, self.f], [self.dq, self.dq], K))

    def ask_without_allocation(self):
        from paper_2112_06188_gb300 import capi

        def call():
            m = self.dq.shape[0]
            oi = torch.full((m, K), -7, dtype=torch.int32, device="cuda")
            od = torch.full((m, K), -7, dtype=torch.int64, device="cuda")
            ptr = lambda t: ctypes.c_void_p(t.data_ptr())
            capi.check(capi.bdl_knn_noalloc(self.f._h, ptr(self.dq), m, K, ptr(oi), ptr(od),
                                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "bdl_knn_noalloc")
            return [(oi, od)]
        return self.run(call)

    def plan(self):
        from paper_2112_06188_gb300.forest import KnnPlan

        def call():
            p = KnnPlan([self.f], [self.dq], K)
            rows = p.launch()
            torch.cuda.synchronize()
            p.close()
            return rows
        return self.run(call)


@pytest.mark.parametrize("dim,split", [(2, "object"), (5, "object"), (3, "spatial")])
def test_one_call_builds_for_those_after_it(dim, split):
    c = Case(dim, split=split)
    assert c.ask() and not c.ask() and not c.ask_without_allocation()
    c.change()
    assert c.ask() and not c.ask_without_allocation()      # more than one call between the last changes
    c.change()
    assert c.ask() and not c.ask_without_allocation()


def test_one_call_per_change_scans():
    c = Case(3)
    assert c.ask()
    for _ in range(3):
        c.change()
        assert not c.ask()
    assert c.ask() and not c.ask()                         # the second and third call of this state
    c.change()
    assert c.ask()                                         # there were three
    c.change()
    assert not c.ask_twice_in_a_batch()                    # one again; a batch is one call
    c.change()
    assert not c.ask()
    assert not c.ask_without_allocation()                  # never builds, but counts
    c.change()
    assert c.ask()
    c.change()
    c.change()                                             # no call in between: as before
    assert not c.ask()
    c.change()
    assert c.plan()
    c.change()
    assert c.ask()                                         # a plan counts as many calls


# on either side of where a scan costs more than the tree: by the buffer's points
# (12 ns each, 24 in 16 dimensions) and by the pairs of query and point in high dimensions
@pytest.mark.parametrize("dim,m,nbuf,builds", [(2, 200, 8_000, False), (2, 200, 15_000, True), (7, 4_000, 2_000, False),
                                               (16, 1_000, 700, False), (16, 4_000, 1_400, True), (10, 40, 14_000, True),
                                               (3, 6_000, 5_000, True)])
def test_scan_where_it_pays(dim, m, nbuf, builds):
    c = Case(dim, m=m, X=16_384, nbuf=nbuf)
    assert c.ask()
    for _ in range(2):
        c.change()
        assert c.ask() == builds
    assert c.ask() != builds
