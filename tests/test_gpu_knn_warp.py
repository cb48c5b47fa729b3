"""The k-NN kernel with one warp per query (small batches, high dimensions)
against brute force, and the thread-per-query kernel (large batches) against
it, bit for bit: every dimension class, leaf sizes from 2 to 64, k at both
ends of its range and at a list longer than the live set, duplicates, erased
points, a part-filled buffer, and leaves far larger than a warp (the spatial
median on duplicates)."""
import numpy as np
import pytest
import torch

from oracle.threads import bruteforce_knn_threads
from paper_2112_06188_gb300 import inputs
from tests.which_kernel import crossing, knn_kernel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_06188_gb300 import build_lib
    build_lib.build()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def forest_of(dim, n, seed, leaf=16, split="object", distinct=0, X=256):
    """A forest after a build, an insert and an erase, and its live points."""
    from paper_2112_06188_gb300.forest import Forest
    draw = (lambda m, s: inputs.duplicate_heavy_points(m, dim, s, distinct)) if distinct else \
           (lambda m, s: inputs.uniform_points(m, dim, s))
    f = Forest(dim, leaf_size=leaf, buffer_size=X, split=split)
    live = inputs.LiveSet(dim)
    for m, s in ((n, seed), (n // 7 + 3, seed + 1)):
        p = draw(m, s)
        f.insert(dev(p))
        live.insert(p)
    gone = inputs.sample_ids(live.live_ids(), len(live.live_ids()) // 9, seed + 2)
    assert f.erase(dev(gone)) == live.erase(gone)
    return f, live


def check(f, live, q, k):
    gi, gd = f.knn(dev(q), k)
    pts, ids = live.live_points()
    bi, bd = bruteforce_knn_threads(pts, ids, q, k)
    assert np.array_equal(gd.cpu().numpy(), bd) and np.array_equal(gi.cpu().numpy(), bi)
    assert f.poll_error() == 0


@pytest.mark.parametrize("dim", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 16])
@pytest.mark.parametrize("k", [1, 10, 32])
def test_dims(dim, k):
    leaf = {1: 8, 10: 16, 32: 64}[k]
    f, live = forest_of(dim, 6_000, 40 * dim + k, leaf=leaf)
    lp, _ = live.live_points()
    q = np.concatenate([inputs.queries_from(lp, 33, 7), inputs.uniform_points(40, dim, 8)])
    check(f, live, q, k)
    check(f, live, q[:1], k)
    # queries off the grid (the C ABI asks for grid points; nothing depends on it)
    check(f, live, q[:5] - (1 << 20), k)
    check(f, live, (q[:5] - (1 << 19)) * 1000, k)


@pytest.mark.parametrize("dim,distinct", [(2, 3), (3, 1), (5, 40)])
@pytest.mark.parametrize("split", ["object", "spatial"])
def test_ties_and_huge_leaves(dim, distinct, split):
    f, live = forest_of(dim, 4_000, 77, split=split, distinct=distinct)
    lp, _ = live.live_points()
    q = np.concatenate([inputs.queries_from(lp, 9, 7), inputs.uniform_points(9, dim, 8)])
    for k in (1, 32):
        check(f, live, q, k)


def test_padding_and_buffer_only():
    for n in (5, 40, 300):
        f, live = forest_of(3, n, 90 + n)
        check(f, live, inputs.uniform_points(7, 3, 5), 32)


def test_deep_trees_with_little_pruning():
    """Leaves of two points in 16 dimensions: the node stack reaches the depth
    from which records are taken one at a time."""
    f, live = forest_of(16, 150_000, 11, leaf=2, X=1024)
    check(f, live, inputs.uniform_points(3, 16, 12), 32)


# on both sides of the batch size from which each dimension takes the thread-per-query
# kernel (k = 1, a small forest), found by asking, and with the launch shapes that kernel has
@pytest.mark.parametrize("dim", [1, 2, 3, 4, 5, 6, 7, 8, 9, 16])
def test_thread_kernel_gives_the_same_rows(dim):
    from paper_2112_06188_gb300.forest import KnnPlan, knn_batch
    f, live = forest_of(dim, 3_000, 60 + dim)
    lp, _ = live.live_points()
    most = 400_000 if dim > 8 else 100_000
    q = dev(np.concatenate([inputs.queries_from(lp, most // 2, 7), inputs.uniform_points(most // 2, dim, 8)]))
    q = q[torch.randperm(most, generator=torch.Generator().manual_seed(1)).cuda()].contiguous()
    c = crossing(f, q, 1)
    q = q[:2 * c + 200].contiguous()
    parts = [knn_kernel(lambda x=x: f.knn(x, 1)) for x in q.split(max(c // 2, 1))]
    assert {name for name, _ in parts} == {"k_knn_warp"}
    wi, wd = (torch.cat(x) for x in zip(*(rows for _, rows in parts)))
    for n, want in ((c, "k_knn_warp"), (c + 1, "k_knn"), (c + 200, "k_knn")):
        name, (gi, gd) = knn_kernel(lambda: f.knn(q[:n], 1))
        assert name == want and torch.equal(gi, wi[:n]) and torch.equal(gd, wd[:n])
    half = q.shape[0] // 2
    name, rows = knn_kernel(lambda: knn_batch([f, f], [q[:half], q[half:]], 1))
    assert name == "k_knn"
    for (gi, gd), want in zip(rows, (slice(0, half), slice(half, None))):
        assert torch.equal(gi, wi[want]) and torch.equal(gd, wd[want])
    if dim in (3, 8, 9):
        for block in (64, 128, 256):
            for per in (32, 64, 128):
                f.set_knn_shape(block, per)
                plan = KnnPlan([f], [q], 1)
                for name, (gi, gd) in (knn_kernel(lambda: f.knn(q, 1)), knn_kernel(lambda: plan.launch()[0])):
                    assert name == "k_knn" and torch.equal(gi, wi) and torch.equal(gd, wd)
                plan.close()
    assert f.poll_error() == 0


# high dimensions at small and large k, with erased points, ties and leaves on either side of 32 points
@pytest.mark.parametrize("dim,k,m", [(8, 16, 300_000), (8, 5, 200_000), (9, 5, 300_000), (11, 5, 300_000), (13, 8, 600_000), (16, 5, 300_000)])
@pytest.mark.parametrize("leaf,distinct", [(16, 0), (40, 50)])
def test_thread_kernel_in_high_dimensions(dim, k, m, leaf, distinct):
    f, live = forest_of(dim, 2_000, 300 + dim, leaf=leaf, distinct=distinct)
    lp, ids = live.live_points()
    few = np.concatenate([inputs.queries_from(lp, 500, 7), inputs.uniform_points(500, dim, 8)])
    q = dev(few).repeat(m // 1_000, 1)
    name, (gi, gd) = knn_kernel(lambda: f.knn(q, k))
    assert name == "k_knn"
    bi, bd = (dev(x) for x in bruteforce_knn_threads(lp, ids, few, k))
    assert torch.equal(gi, bi.repeat(m // 1_000, 1)) and torch.equal(gd, bd.repeat(m // 1_000, 1))
    assert f.poll_error() == 0


@pytest.mark.parametrize("dim,m,k,leaf", [(1, 30_001, 8, 64), (2, 40_003, 5, 33), (3, 70_001, 10, 64), (3, 30_000, 1, 32)])
@pytest.mark.parametrize("distinct", [0, 40])
def test_thread_kernel_with_leaves_over_32_points(dim, m, k, leaf, distinct):
    f, live = forest_of(dim, 9_000, 71 + leaf, leaf=leaf, distinct=distinct)
    lp, _ = live.live_points()
    q = dev(np.concatenate([inputs.queries_from(lp, m // 2, 7), inputs.uniform_points(m - m // 2, dim, 8)]))
    name, (gi, gd) = knn_kernel(lambda: f.knn(q, k))
    assert name == "k_knn" and knn_kernel(lambda: f.knn(q[:5_000], k))[0] == "k_knn_warp"
    for a in range(0, m, 5_000):
        wi, wd = f.knn(q[a:a + 5_000], k)
        assert torch.equal(gi[a:a + 5_000], wi) and torch.equal(gd[a:a + 5_000], wd)
    cnt = torch.zeros(3, dtype=torch.int64, device="cuda")
    ci, cd = f.knn_count(q, k, cnt)
    assert torch.equal(ci, gi) and torch.equal(cd, gd) and f.poll_error() == 0


@pytest.mark.parametrize("dim,n,m,k", [(4, 6_000, 61_003, 32), (7, 20_000, 150_001, 16), (8, 6_000, 60_000, 1),
                                       (10, 3_000, 90_001, 32), (8, 20, 60_100, 32), (8, 40, 60_100, 32)])
@pytest.mark.parametrize("distinct", [0, 7])
def test_queries_in_turn_by_one_warp(dim, n, m, k, distinct):
    """Two to eight queries per warp, each starting with the bound that the
    last one's neighbours give, against one per warp: also with fewer live
    points than k and with points in few places."""
    f, live = forest_of(dim, n, 31 + n, distinct=distinct, X=16)
    lp, _ = live.live_points()
    q = dev(np.concatenate([inputs.queries_from(lp, m // 2, 7), inputs.uniform_points(m - m // 2, dim, 8)]))
    name, (gi, gd) = knn_kernel(lambda: f.knn(q, k))
    assert name == "k_knn_warp"
    for a in range(0, m, 7_000):
        wi, wd = f.knn(q[a:a + 7_000], k)
        assert torch.equal(gi[a:a + 7_000], wi) and torch.equal(gd[a:a + 7_000], wd)
    assert f.poll_error() == 0


@pytest.mark.parametrize("dim,X,n", [(2, 1024, 1023), (3, 64, 5_000), (5, 1024, 20_700), (7, 2048, 33)])
def test_buffer_scanned_first_then_searched(dim, X, n):
    """A forest asked once per update has its buffer scanned by the first small
    call after one, and searched by the calls after it."""
    from paper_2112_06188_gb300.forest import Forest, knn_batch
    f, live = Forest(dim, buffer_size=X), inputs.LiveSet(dim)
    for step, calls in enumerate((1, 1, 3, 3)):
        p = inputs.uniform_points(n if step == 0 else 17, dim, 5 + step)
        f.insert(dev(p))
        live.insert(p)
        if step == 2:
            gone = live.live_ids()[-5:]
            assert f.erase(dev(gone)) == live.erase(gone)
        assert len(f.buffer_ids()) > 0
        lp, ids = live.live_points()
        q = np.concatenate([inputs.queries_from(lp, 20, 1), inputs.uniform_points(13, dim, 2)])
        bi, bd = bruteforce_knn_threads(lp, ids, q, 9)
        for call in range(calls):
            got = [f.knn(dev(q), 9)] if call != 1 else knn_batch([f, f], [dev(q), dev(q)], 9)
            for gi, gd in got:
                assert np.array_equal(gi.cpu().numpy(), bi) and np.array_equal(gd.cpu().numpy(), bd)
    assert f.poll_error() == 0
