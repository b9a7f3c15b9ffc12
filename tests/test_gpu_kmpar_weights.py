"""Weights of many k-means|| candidates: the histogram of the nearest
candidates is counted in shared memory up to 40 960 candidates and in global
memory beyond.  Points on an integer grid, the last 3 000 of them copies of
the first, and an oversampling factor that makes every point off c_0 a
candidate: whole numbers, compared exactly.  And the recluster where its
cluster of CTAs grows, on the same footing."""
import numpy as np
import pytest
import torch

import oracle
import paper_1908_02136_gb300 as kpp
from paper_1908_02136_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [5000, 40960, 40963, 45000])
def test_weights_are_the_histogram_of_the_nearest_candidates(N):
    i = np.arange(N)
    i[N - 3000:] = np.arange(3000)
    x = np.stack([i % 256, i // 256], axis=1).astype(np.float32)
    r = kpp.kmeans_par(torch.from_numpy(x).cuda(), 2, 7, ell=1e13, rounds=1, cand_cap=N)
    cand, w = r["cand"].cpu().numpy(), r["weights"].cpu().numpy()
    assert N - 1 <= cand.size <= N
    first = np.full(N, -1)  # earliest candidate of each grid point
    first[i[cand[::-1]]] = np.arange(cand.size)[::-1]
    lab = first[i]
    assert (lab >= 0).all()
    assert np.array_equal(w, np.bincount(lab, minlength=cand.size))


@pytest.mark.parametrize("N", [300, 301, 2401, 3072, 3073, 4608, 4609])
def test_recluster_at_the_edges_of_its_cluster_sizes(N):
    # a full slice of 384 candidates x 128 features is the most that is staged
    K, d = 6, 128
    x = datagen.integer_points(N, d, seed=N, n_comp=K)
    r = kpp.kmeans_par(torch.from_numpy(x).cuda(), K, 1, ell=1e13, rounds=1, cand_cap=N)
    o = oracle.kmeans_par(x, K, 1e13, 1, 1, 0, cand_cap=N)
    assert r["cand"].numel() == N
    assert np.array_equal(r["cand"].cpu().numpy(), o["cand"])
    assert np.array_equal(r["weights"].cpu().numpy(), o["w"])
    assert np.array_equal(r["idx"].cpu().numpy(), o["idx"])
