"""The screened index builder with fewer than 16 vectors per block on indexes of one to three
nodes: tiles whose other lanes have no edge, tables whose last entry is the allocation's last.
A lane without an edge takes code 0, whatever its stale rows hold.  Codes and edge scalars are
the oracle's bit for bit."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R,d,L,m", [(1, 1, 8, 1, 2), (2, 1, 8, 1, 3), (3, 2, 16, 2, 2), (1, 33, 64, 8, 15),
                                       (2, 32, 64, 1, 7)])
def test_few_nodes_few_vectors(n, R, d, L, m):
    import paper_2402_11354_gb300 as P
    rng = np.random.default_rng(n * 100 + m)
    # a large build first, with infinities, so that the small one finds such rows left in shared memory
    X = rng.standard_normal((4000, d)).astype(np.float32)
    X[::5, 0] = np.inf
    big = rng.integers(0, 4000, size=(4000, 8)).astype(np.int32)
    P.build_codes(P.Graph.from_numpy(big, 0), torch.from_numpy(X).cuda(), L, m, 5).free()
    X = rng.standard_normal((n, d)).astype(np.float32)
    nbrs = np.full((n, R), -1, dtype=np.int32)
    nbrs[:, 0] = rng.integers(0, n, size=n)
    ix = oracle.Index(X, nbrs, 0, L, m, 5)
    codes = P.build_codes(P.Graph.from_numpy(nbrs, 0), torch.from_numpy(X).cuda(), L, m, 5)
    arr = codes.arrays()
    assert np.array_equal(arr["ids"], nbrs)
    valid = nbrs >= 0
    assert np.array_equal(arr["codes"][valid], ix.codes[valid])
    for name, ref in (("enorm", ix.enorm), ("wreg", ix.wreg), ("cres", ix.cres)):
        assert np.array_equal(arr[name].view(np.uint32)[valid], ref.view(np.uint32)[valid]), name
    codes.free()
