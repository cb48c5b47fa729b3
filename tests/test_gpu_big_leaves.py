"""Spatial-median trees whose leaves hold far more points than a warp has
lanes (the rule bounds the depth, not the leaves): erases that find their ids
in such leaves and the leaves' boxes against the oracle, and k-NN by either
kernel (the size of the leaves moves the choice) against the other and, for a
sample, brute force."""
import numpy as np
import pytest
import torch

from oracle.oracle import OracleForest
from oracle.threads import bruteforce_knn_threads, oracle_knn
from paper_2112_06188_gb300 import inputs
from tests.which_kernel import knn_kernel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_06188_gb300 import build_lib
    build_lib.build()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# tight clumps beside uniform points: the clumps of `spread` grid cells end in
# one leaf each (33 .. 8,000 points), the rest in ordinary ones
@pytest.mark.parametrize("dim,clumps,spread", [(2, 1, 1), (2, 5, 8), (3, 40, 2), (2, 600, 1)])
def test_erase_and_boxes(dim, clumps, spread):
    from paper_2112_06188_gb300.forest import Forest
    rng = np.random.default_rng(dim * clumps)
    centre = rng.integers(0, inputs.GRID - spread, size=(clumps, dim))
    near = centre[rng.integers(0, clumps, size=20_000)] + rng.integers(0, spread, size=(20_000, dim))
    pts = np.concatenate([near, rng.integers(0, inputs.GRID, size=(20_000, dim))]).astype(np.int32)
    g, o = Forest(dim, buffer_size=256, split="spatial"), OracleForest(dim, buffer_size=256, split="spatial")
    g.insert(dev(pts))
    o.insert(pts)
    ids = rng.permutation(40_000).astype(np.int32)
    # a list in input order and one in spatial order; repeated and dead ids among them
    for lo, hi in ((0, 1_000), (900, 36_000)):
        e = np.concatenate([ids[lo:hi], ids[lo:lo + 70]])
        assert g.erase(dev(e)) == o.erase(e)
        assert g.poll_error() == 0 and g.size() == o.size() and g.tree_mask() == o.tree_mask()
        for i in g.tree_levels():
            a, b = g.tree(i), o.tree(i)
            assert a["live"] == b["live"] and np.array_equal(a["box"], b["box"])
            assert np.array_equal(a["node_live"], b["node_live"])
            assert set(a["ids"][~a["dead"]].tolist()) == set(b["ids"][~b["dead"]].tolist())
        q = np.concatenate([near[:40], inputs.uniform_points(40, dim, 3)]).astype(np.int32)
        gi, gd = g.knn(dev(q), 7)
        oi, od = oracle_knn(o, q, 7)
        assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gd.cpu().numpy(), od)


@pytest.mark.parametrize("clumps,m", [(5, 150_000), (20_000, 60_000)])
def test_knn_of_skewed_and_even_leaves(clumps, m):
    from paper_2112_06188_gb300.forest import Forest
    rng = np.random.default_rng(clumps)
    centre = rng.integers(0, inputs.GRID, size=(clumps, 2))
    pts = centre[rng.integers(0, clumps, size=20_000)].astype(np.int32)
    f = Forest(2, split="spatial")
    f.insert(dev(pts))
    torch.cuda.synchronize()
    q = inputs.uniform_points(m, 2, 9)
    name, (gi, gd) = knn_kernel(lambda: f.knn(dev(q), 3))
    assert name == "k_knn"
    parts = [knn_kernel(lambda c=c: f.knn(c, 3)) for c in dev(q).split(4_000)]
    assert {name for name, _ in parts} == {"k_knn_warp"}
    wi, wd = (torch.cat(x) for x in zip(*(rows for _, rows in parts)))
    assert torch.equal(gi, wi) and torch.equal(gd, wd)
    bi, bd = bruteforce_knn_threads(pts, np.arange(20_000, dtype=np.int32), q[:300], 3)
    assert np.array_equal(gi[:300].cpu().numpy(), bi) and np.array_equal(gd[:300].cpu().numpy(), bd)
    # leaves of thousands of points move the choice: the same batch on even leaves goes to the other kernel
    name, _ = knn_kernel(lambda: f.knn(dev(q[:35_000]), 3))
    assert name == ("k_knn_warp" if clumps == 5 else "k_knn")
