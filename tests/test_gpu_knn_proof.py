"""How many queries of the exact brute force the tensor-core scores prove: all of them where rows
are well apart, wherever they lie and whatever a few long rows do to the largest norm; none where
more rows are equally near than a list holds, or lie apart by less than the scores' error.  The
results equal the FFMA kernel's bit for bit all the same."""
import pytest
import torch

from test_gpu_knn_exact import P, _check  # noqa: F401

pytestmark = pytest.mark.gpu


# The 10th nearest of 5,000 Gaussian rows and the rows past a list of 26 are 10% apart; the score's
# error is 1e-4 of the product of the norms.
@pytest.mark.parametrize("what", ["plain", "offset", "long row", "two long rows", "offset and a long row"])
def test_proven(P, what):  # noqa: F811
    g = torch.Generator(device="cuda").manual_seed(7)
    n, nq, d, k = 5000, 150, 32, 10
    X = torch.randn(n, d, device="cuda", generator=g)
    Q = torch.randn(nq, d, device="cuda", generator=g)
    if "offset" in what:
        X, Q = X * 0.01 + 100.0, Q * 0.01 + 100.0
    if what == "two long rows":
        X[n // 2] *= 1e12
    if "long row" in what:
        X[0] *= 1e4
    assert P.selftest_knn_left(X, Q, k) == 0
    _check(P, X, Q, k)


def test_left_over(P):  # noqa: F811
    g = torch.Generator(device="cuda").manual_seed(8)
    X = torch.randn(10, 32, device="cuda", generator=g)
    Q = X.repeat(10, 1).contiguous()
    assert P.selftest_knn_left(X.repeat(500, 1).contiguous(), Q, 10) == 100     # every row 500 times
    assert P.selftest_knn_left(X.repeat(200, 1).contiguous(), Q, 10) == -1      # 2,000 rows: the FFMA kernel
    # two groups far apart, the centre in the first: the score's error in the other exceeds its distances
    X = torch.randn(5000, 32, device="cuda", generator=g) * 1e-3
    X[::2] += 1000.0
    assert P.selftest_knn_left(X, X[:64].contiguous(), 10) == 32
    _check(P, X, X[:64].contiguous(), 10)


# norms over six decades, so that rows lie on either side of the norm up to which they matter
@pytest.mark.parametrize("scale", [1.0, 1e-6, 1e8])
def test_mixed_norms(P, scale):  # noqa: F811
    g = torch.Generator(device="cuda").manual_seed(9)
    X = torch.randn(6000, 16, device="cuda", generator=g)
    X *= 10.0 ** (torch.rand(6000, 1, device="cuda", generator=g) * 6 - 3) * scale
    Q = X[::40].clone()
    Q[1::3] *= 1.01
    Q[2::3] = 0.0
    _check(P, X, Q, 12)
