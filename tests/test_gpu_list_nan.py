"""A search whose entry row has an element that is no number: its distance stays at the end of the
list, and the rule by which candidates enter before it keeps the list in order: the candidate of
rank g enters if every one before it did and its distance is below the list's (ef-1-g)-th, which
nothing is where that is no number.  The entry leads to node 1 alone and that to nodes nearer to
the query, so that candidates meet the list [dist, NaN]."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def update(lst, cand, ef):
    """lst: (dist, id) ascending, NaN last."""
    cand = sorted(cand)
    if len(lst) == ef:
        cand = [c for c in cand if c[0] < lst[-1][0]]
    J = 0
    for g, c in enumerate(cand):
        i = ef - 1 - g
        if not (i >= 0 and (i >= len(lst) or c[0] < lst[i][0])):
            break
        J += 1
    return sorted(lst + cand[:J], key=lambda e: (np.isnan(e[0]), e))[:ef]


@pytest.mark.parametrize("ef", [1, 2, 3, 4, 5, 20, 32, 33, 64, 65, 100])
@pytest.mark.parametrize("fan", [3, 20, 32])
def test_entry_without_a_distance(ef, fan):
    import paper_2402_11354_gb300 as P
    n, k = 2 + fan, min(ef, 10)
    X = np.zeros((n, 8), dtype=np.float32)
    X[:, 0] = 100 - np.arange(n)  # node 1 farthest, the others ever nearer
    X[0] = np.nan
    nbrs = np.full((n, 32), -1, dtype=np.int32)
    nbrs[0, 0] = 1
    nbrs[1, :fan] = np.arange(2, n)
    dist = X[:, 0] ** 2
    lst = update([(float("nan"), 0)], [(dist[1], 1)], ef)
    if len(lst) > 1:
        lst = update(lst, [(dist[u], u) for u in range(2, n)], ef)
    ids = [e[1] for e in lst[:k]] + [-1] * (k - len(lst))
    dists = np.array([e[0] for e in lst[:k]] + [np.inf] * (k - len(lst)), dtype=np.float32)
    G, Xt = P.Graph.from_numpy(nbrs, 0), torch.from_numpy(X).cuda()
    codes = P.build_codes(G, Xt, 2, 16, 1)
    Q = torch.zeros(1, 8, device="cuda")
    for routing, mode in ((0, 0), (1, 2)):
        gi, gd = P.search(G, codes, Xt, Q, k, ef, routing=routing, test_mode=mode)[:2]
        assert gi[0].tolist() == ids, routing
        assert np.array_equal(gd[0].cpu().numpy(), dists, equal_nan=True)
