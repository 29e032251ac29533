"""The exact brute force where scores or distances leave FP32's range: a finite query or row
whose products overflow has a score that enters no list, so the lists cannot prove such a
query.  Against the FFMA kernel (pieces of 2,000 rows), bit for bit."""
import pytest
import torch

from test_gpu_knn_exact import P, _check  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["largest queries", "long queries", "long rows", "long rows and queries"])
def test_overflowing_scores(P, what):  # noqa: F811
    g = torch.Generator(device="cuda").manual_seed(23)
    n, nq, d, k = 3000, 140, 32, 10
    X = torch.randn(n, d, device="cuda", generator=g)
    Q = torch.randn(nq, d, device="cuda", generator=g)
    if what == "largest queries":        # BF16 rounds +-3.4e38 to infinity
        Q[::2] = 3.4e38 * torch.sign(Q[::2])
    elif what == "long queries":         # -2 q.x = +inf for every row that is not all zeros
        X = X.abs()
        Q[::3] = -1e38
        Q[1::3] = -1e19
    elif what == "long rows":
        X[::2] *= 1e19
        X[::4] *= 1e18
    elif what == "long rows and queries":
        X[5:] *= 1e18
        Q[::2] *= 1e18
        Q[1::4] *= 1e37
    _check(P, X.contiguous(), Q.contiguous(), k)
