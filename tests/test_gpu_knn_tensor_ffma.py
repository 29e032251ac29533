"""The tensor-core brute force on integer rows against the FFMA kernel itself: pieces of 2,000
rows, below the size from which the exact brute force runs on the tensor cores too."""
import pytest
import torch

import workloads
from test_gpu_knn_exact import P, _pieces  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nq,k", [(3000, 129, 10), (5000, 70, 96), (20_000, 200, 64)])
def test_tensor_against_ffma(P, n, nq, k):  # noqa: F811
    X, Q = workloads.generate(workloads.scaled(workloads.CONFIGS["sift"], n, nq))
    X, Q = torch.from_numpy(X).cuda(), torch.from_numpy(Q).cuda()
    assert P.selftest_knn_left(X[:2000].contiguous(), Q, k) == -1
    ids, dists = P.knn_tensor(X, Q, k)
    ri, rd = _pieces(P, X, Q, k)
    assert torch.equal(ids, ri) and torch.equal(dists, rd)
