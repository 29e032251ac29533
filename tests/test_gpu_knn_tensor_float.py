"""The tensor-core brute force on a million float rows, whose BF16 scores misrank near ties: the
candidates kept per slice of the base absorb that.  20,000 queries make fewer CTAs per query
tile than slices, so lists that followed the CTAs' shares alone would be too few.  Reference:
FP64 distances of the FP32 scores' best rows."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def unit_rows(n, d, latent, seed, clusters):
    """Clustered unit vectors near a subspace, and 20,000 more of them."""
    g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, device="cuda", generator=g)

    centres, image, scales = normal(clusters, latent), normal(latent, d) / math.sqrt(latent), torch.exp(0.75 * normal(d))

    def rows(count):
        z = centres[torch.randint(clusters, (count,), device="cuda", generator=g)] + 0.5 * normal(count, latent)
        y = (z @ image + 0.15 * normal(count, d)) * scales
        return (y / y.norm(dim=1, keepdim=True)).contiguous()

    return rows(n), rows(20_000)


def nearest_f64(X, Q, k):
    sq = (X.double() ** 2).sum(1).float()
    out = torch.empty(len(Q), k, dtype=torch.float64, device="cuda")
    for s in range(0, len(Q), 500):
        q = Q[s:s + 500]
        c = torch.topk(sq - 2.0 * (q @ X.T), k + 64, largest=False).indices
        d = ((X[c].double() - q.double().unsqueeze(1)) ** 2).sum(2)
        out[s:s + 500] = d.sort(1).values[:, :k]
    return out


@pytest.mark.parametrize("n,k,seed", [(1_000_000, 10, 1), (1_000_000, 10, 2), (1_000_000, 96, 3), (300_000, 65, 4)])
def test_a_million_unit_vectors(n, k, seed):
    import paper_2402_11354_gb300 as P
    torch.backends.cuda.matmul.allow_tf32 = False
    X, Q = unit_rows(n, 100, 20, seed, n // 600)
    _, d = P.knn_tensor(X, Q, k)
    ref = nearest_f64(X, Q, k)
    off = (d.double() > ref * (1 + 1e-5) + 1e-6).any(1)
    assert int(off.sum()) == 0
