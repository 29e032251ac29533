"""The exact brute force takes one of two forms by the estimated time; both give the same bits.
One query, a tile's worth and many over bases where the form changes with the number of
queries, the list length or the row length, against each other."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,k,counts", [
    (6_000_000, 64, 100, (1, 33, 600)),   # few queries and long lists on a large base: FFMA; many: scores
    (700_000, 960, 105, (1, 2, 130)),     # the same with long rows
    (2048, 4, 10, (1, 500, 9000)),        # short rows: FFMA
    (65_536, 64, 100, (1, 129, 500)),     # candidates of all segments: 8,192 and 16,384 keys to sort
])
def test_forms_agree(n, d, k, counts):
    import paper_2402_11354_gb300 as P
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.empty(n, d, device="cuda").normal_(generator=g)
    Q = torch.randn(max(counts), d, device="cuda", generator=g)
    ids, dists = P.knn_bruteforce(X, Q, k)
    for c in counts[:-1]:
        ci, cd = P.knn_bruteforce(X, Q[:c].contiguous(), k)
        assert torch.equal(ci, ids[:c]) and torch.equal(cd, dists[:c])
    exact = ((X[ids[:3].long()].double() - Q[:3].double().unsqueeze(1)) ** 2).sum(2)
    assert torch.allclose(dists[:3].double(), exact, rtol=1e-5)
    assert (dists[:, 1:] >= dists[:, :-1]).all()
