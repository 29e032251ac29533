"""Both brute forces on bases where most scores equal the worst kept one: the lowest ids win,
whichever half of a tile they come from.  Integer rows, so that equal rows have equal scores;
the reference ranks by (distance, id)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


# one row throughout; half of the rows zero; two rows in blocks that end inside a tile's halves
@pytest.mark.parametrize("what", ["one row", "half zero", "blocks", "falling"])
@pytest.mark.parametrize("n,nq,k", [(2048, 3, 1), (5000, 129, 26), (40_000, 300, 96)])
def test_lowest_ids_win(what, n, nq, k):
    import paper_2402_11354_gb300 as P
    d = 16
    g = torch.Generator(device="cuda").manual_seed(n + k)
    X = torch.randint(0, 4, (n, d), device="cuda", generator=g).float()
    Q = torch.randint(0, 4, (nq, d), device="cuda", generator=g).float()
    i = torch.arange(n, device="cuda")
    if what == "one row":
        X[:] = X[0]
    elif what == "half zero":
        X[::2] = 0.0
        Q[::2] = 0.0
    elif what == "blocks":
        X = X[(i // 100) % 2].contiguous()
    elif what == "falling":  # ever nearer to the query: every row enters, then a run of ties
        X[:] = 0.0
        X[:, 0] = (200 - i * 200 // n).float()
        Q[:] = 0.0
    D = (Q * Q).sum(1, keepdim=True) + (X * X).sum(1) - 2.0 * (Q @ X.T)  # exact integers
    key, _ = torch.sort(D.long() * n + i, dim=1)
    ids, dists = (key[:, :k] % n).int(), (key[:, :k] // n).float()
    for fn in (P.knn_tensor, P.knn_bruteforce):
        gi, gd = fn(X, Q, k)
        assert torch.equal(gi, ids) and torch.equal(gd, dists), fn.__name__
