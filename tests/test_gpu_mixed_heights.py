"""Batched builds of trees of several heights, where a depth nearer the roots
holds more nodes than a deeper one: the boxes of every tree, and no depth of
many nodes left to one block (one taller tree beside 500 must not make the
box pass many times as long)."""
import numpy as np
import pytest
import torch

from paper_2112_06188_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_06188_gb300 import build_lib
    build_lib.build()


def box_pass(split, sizes, kernel, check=False):
    """ms of `kernel` (the least of three builds) for forests of these sizes built together."""
    from paper_2112_06188_gb300 import capi
    from paper_2112_06188_gb300.forest import Forest, insert_batch
    pts = [inputs.uniform_points(n, 2, seed=n + j) for j, n in enumerate(sizes)]
    dev = [torch.from_numpy(p).cuda() for p in pts]
    best = 1e9
    for _ in range(3):
        fs = [Forest(2, split=split) for _ in sizes]
        torch.cuda.synchronize()
        capi.bdl_profile(1)
        insert_batch(fs, dev)
        torch.cuda.synchronize()
        best = min(best, capi.bdl_profile_read_bytes()[kernel][0])
        capi.bdl_profile(0)
        if check:
            check = False
            for f, p in list(zip(fs, pts))[:40]:
                assert f.poll_error() == 0
                for lv in f.tree_levels():
                    t = f.tree(lv)
                    x = p[t["ids"]]
                    root = t["box"][0]
                    assert np.array_equal(root, np.concatenate([x.min(0), x.max(0)])) and t["node_live"][0] == len(x)
                    inner = np.flatnonzero(t["child"][:, 0] >= 0)
                    a, b = t["box"][t["child"][inner, 0]], t["box"][t["child"][inner, 1]]
                    assert np.array_equal(t["box"][inner, :2], np.minimum(a[:, :2], b[:, :2]))
                    assert np.array_equal(t["box"][inner, 2:], np.maximum(a[:, 2:], b[:, 2:]))
        for f in fs:
            f.close()
    return best


@pytest.mark.parametrize("split,kernel,tall,low", [("spatial", "k_sp_box", 20_000, 9_000),
                                                   ("object", "k_build_finish", 60_000, 30_000)])
def test_one_taller_tree_among_many(split, kernel, tall, low):
    n = 500 if split == "spatial" else 300
    even = box_pass(split, [tall] * (n + 1), kernel)
    mixed = box_pass(split, [tall] + [low] * n, kernel, check=True)
    assert mixed < 4 * even + 0.1
