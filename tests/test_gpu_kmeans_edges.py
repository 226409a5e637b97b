"""k-means where its kernels' tiling can go wrong: the assignment's pairs of
points (128 apart, blocks of 256) and groups of four centroids, the update's
lanes of 16 labels, warps of 512 and chunks of 4,096, label arrays off the wide
loads' alignment, clusters of no point and of all of them.  Labels and centroids
are decided in stated precisions, so they equal the oracle's bit for bit."""
import numpy as np
import pytest
import torch

import oracle
import paper_1512_06473_gb300 as q
import synth

pytestmark = pytest.mark.gpu


def run(pts, init, iters):
    D, a = q.kmeans(torch.from_numpy(pts).cuda(), torch.from_numpy(init).cuda(), iters)
    D, a = D.cpu().numpy(), a.cpu().numpy()
    for m in range(len(pts)):
        cen, am = oracle.kmeans(pts[m], init[m], iters)
        assert np.array_equal(a[m], am), m
        assert np.array_equal(D[m], cen), m


@pytest.mark.parametrize("M,P,Csp,K", [
    (1, 1, 1, 1), (3, 15, 2, 4), (2, 16, 3, 5), (2, 128, 4, 6), (3, 129, 5, 7), (2, 256, 8, 8),
    (3, 257, 4, 9), (2, 511, 7, 17), (2, 513, 4, 256), (1, 4096, 4, 33), (2, 4097, 6, 128),
    (3, 9001, 4, 12),
])
def test_sizes(M, P, Csp, K):
    pts = synth.normal((M, P, Csp), 1.0, 500 + P)
    init = synth.normal((M, K, Csp), 1.0, 501 + K)
    run(pts, init, 3)


@pytest.mark.parametrize("P", [700, 5000])
def test_one_cluster_takes_all(P):
    pts = synth.normal((2, P, 4), 1.0, 7)
    init = np.full((2, 5, 4), 1e3, np.float32)
    init[:, 3] = 0.0
    run(pts, init, 2)
