"""The list update at the list lengths where its form changes (slots in one or two registers'
worth of lanes, more than 64 slots, a partial last group), on rows of small integers: equal
distances everywhere, repeated rows, a node listed twice.  Distances are exact, so plain
routing and PEOs with every edge passing (test_mode 2) both equal the oracle's plain search
bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from workloads.graph import build_graph

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    import paper_2402_11354_gb300 as P
    P.load()
    rng = np.random.default_rng(5)
    X = rng.integers(0, 4, size=(1500, 8)).astype(np.float32)
    X[700:900] = X[:200]
    Q = rng.integers(0, 4, size=(120, 8)).astype(np.float32)
    out = {}
    for R in (32, 48):
        nbrs, entry = build_graph(X, R)
        nbrs[::7, -1] = nbrs[::7, 0]  # the first neighbour once more in the last slot
        G = P.Graph.from_numpy(nbrs, entry)
        Xt = torch.from_numpy(X).cuda()
        out[R] = (P, G, Xt, torch.from_numpy(Q).cuda(), P.build_codes(G, Xt, 4, 16, 9),
                  oracle.Index(X, nbrs, entry, 4, 16, 9), Q)
    return out


@pytest.mark.parametrize("R", [32, 48])
@pytest.mark.parametrize("ef", [1, 2, 31, 32, 33, 63, 64, 65, 96, 97, 129, 500, 1024])
def test_equals_the_oracle(case, R, ef):
    P, G, X, Q, codes, ix, Qh = case[R]
    k = min(ef, 10)
    ref = ix.search(Qh, k, ef, routing=0)
    for routing, mode in ((0, 0), (1, 2)):
        for gather in (4, 8):
            ids, dists, cnt = P.search(G, codes, X, Q, k, ef, routing=routing, test_mode=mode, counters=True,
                                       gather_rows=gather)
            assert np.array_equal(ids.cpu().numpy(), ref["ids"]), (routing, gather)
            assert np.array_equal(dists.cpu().numpy(), ref["dists"])
            assert np.array_equal(cnt.cpu().numpy()[:, 0], ref["counters"][:, 0])  # expansions
