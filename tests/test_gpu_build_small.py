"""Builds small enough that their subtrees leave SMs idle take one more global
level: every tree equals the oracle's on both sides of the sizes where that
begins (6,144 records in a subtree) and at odd sizes."""
import numpy as np
import pytest
import torch

from oracle.oracle import OracleForest
from paper_2112_06188_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_06188_gb300 import build_lib
    build_lib.build()


@pytest.mark.parametrize("dim", [1, 2, 3, 5])
@pytest.mark.parametrize("X,n", [(4_097, 4_097), (6_143, 6_143), (6_145, 6_145), (6_147, 12_300), (8_191, 8_191),
                                 (8_193, 8_193), (12_289, 24_600), (1_024, 8_192), (1_024, 30_011)])
def test_trees(dim, X, n):
    from paper_2112_06188_gb300.forest import Forest
    pts = inputs.uniform_points(n, dim, seed=n + dim)
    pts[: n // 3, 0] = pts[0, 0]          # ties across the tiles in one coordinate
    g, o = Forest(dim, buffer_size=X), OracleForest(dim, buffer_size=X)
    g.insert(torch.from_numpy(pts).cuda())
    o.insert(pts)
    assert g.poll_error() == 0 and g.tree_mask() == o.tree_mask() != 0
    for i in g.tree_levels():
        a, b = g.tree(i), o.tree(i)
        for what in ("key", "child", "box", "node_live", "leaf_off"):
            assert np.array_equal(a[what], b[what]), what
        for lo, hi in zip(a["leaf_off"][:-1], a["leaf_off"][1:]):
            assert set(a["ids"][lo:hi].tolist()) == set(b["ids"][lo:hi].tolist())
