"""Spatial-median builds with more records than one pass of the resident
blocks takes (about 233,000 on 152 SMs), so that blocks go round several
times per level: trees of several heights in one build, and clustered points,
against the oracle node by node."""
import numpy as np
import pytest
import torch

from oracle.oracle import OracleForest, bruteforce_knn
from paper_2112_06188_gb300 import inputs
from tests.test_gpu_parity import assert_same_forest, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,L,X,gen", [(2, 600_003, 16, 1024, "uniform"), (3, 300_001, 4, 64, "uniform"),
                                           (2, 500_000, 16, 512, "clusters"), (5, 262_144, 32, 256, "uniform")])
def test_blocks_go_round(dim, n, L, X, gen):
    from paper_2112_06188_gb300 import build_lib
    from paper_2112_06188_gb300.forest import Forest
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build_lib.build()
    draw = inputs.gaussian_clusters if gen == "clusters" else inputs.uniform_points
    pts = draw(n, dim, 17)
    g = Forest(dim, leaf_size=L, buffer_size=X, split="spatial")
    o = OracleForest(dim, leaf_size=L, buffer_size=X, split="spatial")
    assert np.array_equal(g.insert(to_dev(pts)).cpu().numpy(), o.insert(pts))
    assert_same_forest(g, o)
    q = pts[::n // 5]
    gi, gd = g.knn(to_dev(q), 7)
    bi, bd = bruteforce_knn(pts, np.arange(n, dtype=np.int32), q, 7)
    assert np.array_equal(gd.cpu().numpy(), bd) and np.array_equal(gi.cpu().numpy(), bi)
    assert g.poll_error() == 0
