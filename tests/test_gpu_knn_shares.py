"""The tensor-core brute force where the work goes to the CTAs by whole slices of the base for rows
whose scores are rounded and by equal shares for integer rows: more CTAs for the latter (53 query
tiles, two slices each), as many (93 tiles, three slices), and slices alone (one query tile).
Integer rows against keys of exact distances; the same rows divided by three, which BF16 rounds,
against the exact brute force."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nq,k", [(314_253, 6_681, 1), (605_982, 11_863, 1), (150_001, 127, 3)])
def test_shares(n, nq, k):
    import paper_2402_11354_gb300 as P
    d = 12
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randint(0, 30, (n, d), device="cuda", generator=g).float()
    Q = torch.randint(0, 30, (nq, d), device="cuda", generator=g).float()
    ids, dists = P.knn_tensor(X, Q, k)
    x2, i = (X * X).sum(1), torch.arange(n, device="cuda")
    for s in range(0, nq, 200):
        q = Q[s:s + 200]
        D = (q * q).sum(1, keepdim=True) + x2 - 2.0 * (q @ X.T)  # exact integers
        key = torch.topk(D.long() * n + i, k, largest=False).values.sort(1).values
        assert torch.equal(ids[s:s + 200].long(), key % n) and torch.equal(dists[s:s + 200].long(), key // n)
    X, Q = X / 3.0, Q / 3.0
    ids, dists = P.knn_tensor(X, Q, k)
    _, exact = P.knn_bruteforce(X, Q, k)
    # the k best scores lie within twice the scores' error, 4.1 2^-8 of the norms, of the k nearest
    err = 4.1 * 2.0 ** -8 * X.norm(dim=1).max() * Q.norm(dim=1, keepdim=True)
    assert (dists <= exact * (1 + 1e-5) + 2 * err).all() and (dists >= exact * (1 - 1e-5)).all()
