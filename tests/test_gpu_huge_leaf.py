"""Spatial-median trees with leaves of millions of points in one place (the
rule bounds the depth, not the leaves): every leaf's box and live count equals
its points', no barrier gives up, and no warp goes through such a leaf alone
while the other blocks wait (8M points by one warp take more than 100 ms)."""
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


def boxes_from_points(pts, leaf_off):
    """Per leaf the extent of its points (rows in leaf order), empty leaves the empty box."""
    nl, d = len(leaf_off) - 1, pts.shape[1]
    box = np.empty((nl, 2 * d), np.int32)
    box[:, :d], box[:, d:] = np.iinfo(np.int32).max, np.iinfo(np.int32).min
    full = np.flatnonzero(np.diff(leaf_off) > 0)
    box[full, :d] = np.minimum.reduceat(pts, leaf_off[full], axis=0)
    box[full, d:] = np.maximum.reduceat(pts, leaf_off[full], axis=0)
    return box


# clumps of `spread` grid cells with `sizes` points each, on both sides of the size from which
# a leaf is dealt to all warps (8,192 points), beside 60,000 uniform points
@pytest.mark.parametrize("dim,sizes,spread", [(3, [8_000_000], 1), (2, [3_000_000, 700_001, 8_193, 8_192, 8_191], 1),
                                              (16, [400_003, 20_000], 1), (5, [50_000] * 30, 3), (1, [1_000_000], 2)])
def test_boxes(dim, sizes, spread):
    from paper_2112_06188_gb300 import capi
    from paper_2112_06188_gb300.forest import Forest
    rng = np.random.default_rng(dim)
    parts = [inputs.uniform_points(60_000, dim, 5)]
    for m in sizes:
        parts.append(rng.integers(0, inputs.GRID - spread, size=dim) + rng.integers(0, spread, size=(m, dim)))
    pts = np.concatenate(parts).astype(np.int32)
    pts = pts[rng.permutation(len(pts))]
    dev = torch.from_numpy(pts).cuda()
    f = Forest(dim, split="spatial")
    f.insert(dev[:100_000])          # (the first build of a process loads the kernels)
    f.close()
    f = Forest(dim, split="spatial", buffer_size=16_384)
    torch.cuda.synchronize()
    capi.bdl_profile(1)
    f.insert(dev)
    torch.cuda.synchronize()
    ms = capi.bdl_profile_read_bytes()["k_sp_box"][0]
    capi.bdl_profile(0)
    assert f.poll_error() == 0
    assert ms < 30
    for lv in f.tree_levels():
        t = f.tree(lv)
        h, d = t["h"], dim
        # slots of a level's nodes in order, from the root down
        at = np.zeros(1, np.int64)
        levels = [at]
        for _ in range(h):
            at = t["child"][at].reshape(-1).astype(np.int64)
            levels.append(at)
        assert np.array_equal(-1 - t["child"][at, 0], np.arange(1 << h))
        box = boxes_from_points(pts[t["ids"]], t["leaf_off"])
        live = np.diff(t["leaf_off"])
        for at in reversed(levels):
            assert np.array_equal(t["box"][at], box) and np.array_equal(t["node_live"][at], live)
            if len(at) > 1:
                box = np.concatenate([np.minimum(box[0::2, :d], box[1::2, :d]), np.maximum(box[0::2, d:], box[1::2, d:])], 1)
                live = live[0::2] + live[1::2]
    f.close()
