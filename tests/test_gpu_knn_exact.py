"""The exact brute force on bases large enough for the tensor-core scores (two-term BF16 with
a proof per query, the FFMA kernel for the rest) against the FFMA kernel alone: the same
base in pieces of 2,000 rows, which the FFMA kernel takes, merged by (distance, id).  Both
form the same FP32 sums, so ids and distances are equal bit for bit, on every input: near
ties, repeated rows (more equal distances than a list has room for), rows and queries of
zeros, huge, tiny and non-finite values."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2402_11354_gb300 as P
    P.load()
    return P


def _pieces(P, X, Q, k, step=2000):
    keys = []
    for s in range(0, len(X), step):
        x = X[s:s + step].contiguous()
        i, d = P.knn_bruteforce(x, Q, k)
        key = (d.view(torch.int32).long() << 32) | (i.long() + s)
        keys.append(torch.where(i < 0, torch.full_like(key, 2 ** 63 - 1), key))
    best = torch.sort(torch.cat(keys, 1), 1).values[:, :k]
    none = best == 2 ** 63 - 1
    ids = torch.where(none, -1, (best & 0xFFFFFFFF)).int()
    dists = torch.where(none, float("inf"), (best >> 32).int().view(torch.float32))
    return ids, dists


def _check(P, X, Q, k):
    ids, dists = P.knn_bruteforce(X, Q, k)
    ri, rd = _pieces(P, X, Q, k)
    assert torch.equal(ids, ri)
    assert torch.equal(dists.view(torch.int32), rd.view(torch.int32))


# sizes around a tile (256 rows, 128 queries), the smallest base the scores take, lists up to
# the longest (k = 105) and beyond (FFMA alone)
@pytest.mark.parametrize("n,nq,d,k", [(2048, 1, 4, 1), (2049, 127, 64, 10), (4095, 129, 100, 33), (5000, 128, 68, 97),
                                      (20_000, 300, 128, 105), (3000, 40, 96, 106), (6000, 17, 960, 20),
                                      (2500, 5, 2048, 105)])
def test_random_rows(P, n, nq, d, k):
    g = torch.Generator(device="cuda").manual_seed(n + d)
    X = torch.randn(n, d, device="cuda", generator=g)
    Q = torch.randn(nq, d, device="cuda", generator=g)
    Q[: nq // 2] = X[: nq // 2] + 0.01 * Q[: nq // 2]
    _check(P, X, Q, k)


@pytest.mark.parametrize("what", ["repeated", "offset", "zeros", "huge", "tiny", "mixed", "nan", "inf", "zero query"])
def test_hard_values(P, what):
    g = torch.Generator(device="cuda").manual_seed(11)
    n, nq, d, k = 5000, 150, 32, 10
    X = torch.randn(n, d, device="cuda", generator=g)
    Q = torch.randn(nq, d, device="cuda", generator=g)
    if what == "repeated":      # 100 distinct rows, each 50 times: ties far beyond a list's slack
        X = X[:100].repeat(50, 1).contiguous()
        Q = X[:nq].clone()
    elif what == "offset":      # far from the origin: the scores' error exceeds the distances
        X, Q = X * 0.01 + 1000.0, Q * 0.01 + 1000.0
    elif what == "zeros":
        X[::2] = 0.0
    elif what == "huge":
        X, Q = X * 1e18, Q * 1e18
    elif what == "tiny":
        X, Q = X * 1e-20, Q * 1e-20
    elif what == "mixed":
        X[::3] *= 1e-15
        X[1::3] *= 1e6
    elif what == "nan":
        X[17, 3] = float("nan")
        Q[5, 1] = float("nan")
    elif what == "inf":
        X[17, 3] = float("inf")
        Q[5, 1] = -float("inf")
    elif what == "zero query":
        Q[:] = 0.0
    _check(P, X.contiguous(), Q.contiguous(), k)


def test_base_converted_in_slabs(P):
    """More than 1 GiB of converted rows: the base is taken in two slabs."""
    g = torch.Generator(device="cuda").manual_seed(3)
    X = torch.randn(140_000, 2048, device="cuda", generator=g)
    Q = X[::7000][:20] + 0.05 * torch.randn(20, 2048, device="cuda", generator=g)
    ids, dists = P.knn_bruteforce(X, Q.contiguous(), 7)
    ri, rd = _pieces(P, X, Q.contiguous(), 7)
    assert torch.equal(ids, ri) and torch.equal(dists, rd)
