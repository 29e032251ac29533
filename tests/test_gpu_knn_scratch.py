"""The exact brute force's scratch stays within the 1 GiB that its header states, whatever the
number of queries and the size of the base, and slicing changes no result."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu

USED_MEM_HIGH = 8  # CU_MEMPOOL_ATTR_USED_MEM_HIGH


def _pool():
    cu = ctypes.CDLL("libcuda.so.1")
    torch.zeros(1, device="cuda")
    dev, pool = ctypes.c_int(), ctypes.c_void_p()
    assert cu.cuDeviceGet(ctypes.byref(dev), torch.cuda.current_device()) == 0
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), dev) == 0
    return cu, pool


# many queries (their converted rows alone exceed the bound; a last slice of one query), many
# rows (several slabs), long lists of few slices
@pytest.mark.parametrize("n,nq,d,k", [(20_000, 320_001, 960, 10), (2_000_000, 3000, 128, 10), (20_000, 300_000, 64, 105)])
def test_scratch_bound(n, nq, d, k):
    import paper_2402_11354_gb300 as P
    g = torch.Generator(device="cuda").manual_seed(n + k)
    X = torch.randn(n, d, device="cuda", generator=g)
    Q = torch.randn(nq, d, device="cuda", generator=g)
    P.knn_bruteforce(X[:3000].contiguous(), Q[:10].contiguous(), 1)
    torch.cuda.synchronize()
    cu, pool = _pool()
    value = ctypes.c_uint64(0)
    assert cu.cuMemPoolSetAttribute(pool, USED_MEM_HIGH, ctypes.byref(value)) == 0
    ids, dists = P.knn_bruteforce(X, Q, k)
    torch.cuda.synchronize()
    assert cu.cuMemPoolGetAttribute(pool, USED_MEM_HIGH, ctypes.byref(value)) == 0
    assert 0 < value.value <= 1.01 * 2 ** 30
    pick = torch.cat([torch.arange(0, nq, nq // 50, device="cuda"), torch.tensor([nq - 1], device="cuda")])
    pi, pd = P.knn_bruteforce(X, Q[pick].contiguous(), k)
    assert torch.equal(ids[pick], pi) and torch.equal(dists[pick], pd)


def test_left_over_queries_in_slices():
    """Rows that the scores cannot tell apart: every query is left to the FFMA kernel, whose
    lists (129 chunks of 105 keys each) take 9,888 queries at a time."""
    import paper_2402_11354_gb300 as P
    g = torch.Generator(device="cuda").manual_seed(9)
    X = torch.randint(0, 2, (2_100_000, 4), device="cuda", generator=g).float()
    Q = torch.randint(0, 2, (12_000, 4), device="cuda", generator=g).float()
    k = 105
    ids, dists = P.knn_bruteforce(X, Q, k)
    i = torch.arange(len(X), device="cuda")
    code = (X * torch.tensor([1.0, 2.0, 4.0, 8.0], device="cuda")).sum(1)
    want = (Q * torch.tensor([1.0, 2.0, 4.0, 8.0], device="cuda")).sum(1)
    for c in range(16):  # the k lowest ids among the rows that equal the query
        rows = i[code == c][:k].int()
        assert torch.equal(ids[want == c], rows.expand(int((want == c).sum()), k))
    assert not dists.any()
