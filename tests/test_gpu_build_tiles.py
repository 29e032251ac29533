"""The tiled index builder (up to 16 vectors per block) at the sizes where a tile, a block
or a staged chunk ends: every record and table against the oracle.  Codes, ||e||, w_reg and
sqrt(L) w_res are the same sums in the same order on both sides, so they are equal bit for
bit; node tables and node terms agree within 1e-5 of the magnitude of their terms."""
import numpy as np
import pytest
import torch

import oracle
import parity

pytestmark = pytest.mark.gpu


def _graph(rng, n, R, fill):
    nbrs = rng.integers(0, n, size=(n, R)).astype(np.int32)
    nbrs[rng.random((n, R)) >= fill] = -1
    return nbrs


# block lengths 1, 2, 3, 4, 5, 10, 16, 40 and 320 (one block); coordinates staged in part; fewer
# than 16 vectors; out-degrees 1, 33 and 64; one node, one edge, tiles with one edge left over
@pytest.mark.parametrize("n,R,d,L,m,fill,perm", [
    (1, 1, 4, 1, 16, 1.0, False),
    (65, 1, 128, 8, 16, 1.0, False),
    (129, 64, 128, 8, 16, 0.5, False),
    (300, 33, 100, 10, 16, 0.3, True),
    (257, 32, 36, 12, 16, 0.9, False),
    (130, 32, 40, 8, 5, 0.6, True),
    (200, 7, 12, 12, 2, 0.8, False),
    (150, 32, 28, 14, 9, 0.0, False),
    (97, 16, 960, 24, 16, 0.7, False),
    (90, 16, 320, 1, 11, 0.7, True),
    # blocks of 8..64 coordinates, a multiple of 4: estimates on the tensor cores settle most codes
    (1, 1, 8, 1, 16, 1.0, False),
    (500, 32, 128, 8, 16, 0.4, True),
    (300, 20, 96, 8, 16, 0.8, False),
    (200, 64, 64, 8, 7, 0.9, False),
    (150, 33, 64, 1, 16, 0.5, False),
    (260, 9, 240, 5, 16, 1.0, False),
    (120, 32, 960, 24, 16, 0.6, True),
    (400, 16, 280, 35, 16, 0.9, False),
])
def test_records_and_tables(n, R, d, L, m, fill, perm):
    import paper_2402_11354_gb300 as P
    rng = np.random.default_rng(n * 1000 + d)
    X = rng.standard_normal((n, d)).astype(np.float32)
    X[n // 2] = X[0]                    # duplicate vectors: degenerate edges
    X[:, : d // L] *= (rng.random((n, 1)) < 0.5)  # zero blocks
    nbrs = _graph(rng, n, R, fill)
    nbrs[0, 0] = n // 2
    p = rng.permutation(d).astype(np.int32) if perm else None
    ix = oracle.Index(X, nbrs, 0, L, m, 77, perm=p)
    codes = P.build_codes(P.Graph.from_numpy(nbrs, 0), torch.from_numpy(X).cuda(), L, m, 77,
                          perm=torch.from_numpy(p).cuda() if perm else None)
    arr = codes.arrays()
    assert np.array_equal(arr["ids"], nbrs)
    valid = nbrs >= 0
    for name, ref in (("enorm", ix.enorm), ("wreg", ix.wreg), ("cres", ix.cres)):
        assert np.array_equal(arr[name].view(np.uint32)[valid], ref.view(np.uint32)[valid]), name
        assert not arr[name][~valid].any()
    assert np.array_equal(arr["codes"][valid], ix.codes[valid])
    Xi = (X[:, p] if perm else X).astype(np.float64)
    t = np.concatenate([(Xi @ ix.B.astype(np.float64).T)[:, None, :],
                        np.einsum("nlk,ljk->nlj", Xi.reshape(n, L, d // L), ix.A.astype(np.float64))], axis=1)
    scale = np.linalg.norm(Xi, axis=1)[:, None, None] * np.concatenate(
        [np.linalg.norm(ix.B, axis=1)[None], np.linalg.norm(ix.A, axis=2)], axis=0)[None]
    assert np.all(parity.close(arr["tv"], t, scale))
    sv, sv_scale = parity.node_terms(t, np.where(valid[:, :, None], ix.codes, 0), ix.wreg, ix.cres)
    assert np.all(parity.close(arr["sv"], sv, sv_scale)[valid])
    codes.free()


@pytest.mark.parametrize("what", ["integer", "equal vectors' sums", "tiny", "huge", "mixed", "nan"])
def test_codes_of_hard_values(what):
    """Sums that tie, vanish, overflow or are not numbers: the estimates settle nothing wrong."""
    import paper_2402_11354_gb300 as P
    rng = np.random.default_rng(4)
    n, R, d, L, m = 300, 12, 64, 4, 16
    X = rng.standard_normal((n, d)).astype(np.float32)
    if what == "integer":
        X = rng.integers(0, 3, size=(n, d)).astype(np.float32)
    elif what == "equal vectors' sums":  # one coordinate per block: |sums| are multiples of one another
        X[:] = 0.0
        X[np.arange(n), rng.integers(0, d, n)] = 1.0
    elif what == "tiny":
        X *= np.float32(1e-18)
        X[::2] *= np.float32(1e-12)
    elif what == "huge":
        X *= np.float32(1e18)
        X[::3] *= np.float32(1e3)
    elif what == "mixed":
        X *= (10.0 ** rng.uniform(-18, 18, size=(n, d))).astype(np.float32)
    elif what == "nan":
        X[5, 7] = np.nan
        X[9, 40] = np.inf
    nbrs = _graph(rng, n, R, 0.9)
    with np.errstate(all="ignore"):
        ix = oracle.Index(X, nbrs, 0, L, m, 3)
    codes = P.build_codes(P.Graph.from_numpy(nbrs, 0), torch.from_numpy(X).cuda(), L, m, 3)
    arr = codes.arrays()
    valid = nbrs >= 0
    assert np.array_equal(arr["codes"][valid], ix.codes[valid])
    for name, ref in (("enorm", ix.enorm), ("wreg", ix.wreg), ("cres", ix.cres)):
        assert np.array_equal(np.nan_to_num(arr[name][valid], nan=-1), np.nan_to_num(ref[valid], nan=-1)), name
    codes.free()
