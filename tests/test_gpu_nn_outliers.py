"""Nearest neighbours where the search leaves the first ring of cells: a few
centres far from a dense cluster (the warp finishes those together), bit
exact against the oracle."""
import numpy as np
import pytest

import gemtest as gt
import oracle
from paper_2509_25075_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 5, 16])
@pytest.mark.parametrize("M,far", [(2, 1), (20, 3), (33, 32), (700, 40), (3000, 7), (3000, 300)])
def test_far_centres(M, far, k):
    rng = np.random.default_rng(M + far)
    th = syn.gaussians(syn.Workload("far", d=64, M=M, B=1, n_clusters=1, seed=3))
    th[:, 0:3] = rng.normal(scale=1.0, size=(M, 3))
    th[:far, 0:3] = rng.uniform(-60, 60, size=(far, 3))
    th[far // 2, 0:3] = th[M - 1, 0:3]  # a pair at distance zero
    ctx = gt.context(syn.Workload("far", d=32, M=M, B=1, seed=1))
    dist, idx = ctx.gem_nn_distance(gt.to_dev(th), k)
    rd, ri = oracle.nn_distance(th[:, 0:3], k)
    np.testing.assert_array_equal(idx.cpu().numpy(), ri)
    np.testing.assert_array_equal(dist.cpu().numpy(), np.asarray(rd, dtype=np.float32))
    ctx.close()


@pytest.mark.parametrize("k", [1, 3, 4, 8, 16])
@pytest.mark.parametrize("shape", ["plane", "line", "lattice", "uniform", "pair of heaps"])
@pytest.mark.parametrize("M", [17, 1000, 5000])
def test_centres_that_need_many_rings(M, shape, k):
    """Sets where whole warps go on beyond the first ring (k neighbours, flat
    and linear sets), with ties and empty cells."""
    rng = np.random.default_rng(M + k)
    p = rng.uniform(-50, 50, (M, 3))
    if shape == "plane":
        p[:, rng.integers(3)] = 1.5
    elif shape == "line":
        p[:, 1:] = 0.0
    elif shape == "lattice":
        p = rng.integers(-8, 9, (M, 3)).astype(float)
    elif shape == "pair of heaps":
        p = rng.normal(size=(M, 3)) * 0.3 + np.where(np.arange(M) % 9 == 0, 50.0, -50.0)[:, None]
    th = syn.gaussians(syn.Workload("far", d=64, M=M, B=1, n_clusters=1, seed=3))
    th[:, 0:3] = p
    ctx = gt.context(syn.Workload("far", d=32, M=M, B=1, seed=1))
    dist, idx = ctx.gem_nn_distance(gt.to_dev(th), k)
    rd, ri = oracle.nn_distance(th[:, 0:3], k)
    np.testing.assert_array_equal(idx.cpu().numpy(), ri)
    np.testing.assert_array_equal(dist.cpu().numpy(), np.asarray(rd, dtype=np.float32))
    ctx.close()
