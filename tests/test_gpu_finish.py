"""The block-wide selection that ends a search of many splits: one block's worth of entries, several
groups of splits, and more equal scores than it keeps."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


# 1 and 37 queries: a block has the SM's shared memory; 300: two groups of splits; 512: one
@pytest.mark.parametrize("nq", [1, 37, 300, 512])
@pytest.mark.parametrize("ng,topk,copies", [(60000, 100, 0), (60000, 20, 0), (9001, 100, 0), (40000, 100, 3000),
                                            (40000, 15, 3000), (40000, 40, 700)])
def test_top_k_of_many_splits(nq, ng, topk, copies):
    """Exact top-K against FP64: the distances of the K nearest, in order, within 1e-5 (FP32 dot
    products of 128 terms, 2^-24 each), and every index at its distance. Copies of one gallery row,
    nearest to all queries, come first and by index."""
    import paper_2306_08792_gb300 as gcr
    g = torch.Generator(device="cuda").manual_seed(nq + ng + topk)
    q = torch.randn(nq, 128, generator=g, device="cuda")
    b = torch.randn(ng, 128, generator=g, device="cuda")
    where = torch.randperm(ng, generator=g, device="cuda")[:copies].sort().values
    if copies:
        q = q[:1] + 0.01 * q
        b[where] = q[:1]
    q, b = gcr.gcr_normalize(q), gcr.gcr_normalize(b)
    idx, dist = gcr.gcr_rerank(q, b, gcr.default_params(precision="tf32", topk_out=topk))
    D = 2.0 - 2.0 * (q.double() @ b.double().T)
    want = D.topk(topk, dim=1, largest=False).values
    got = D.gather(1, idx.long())
    assert (got - want).abs().max() < 1e-5 and (dist.double() - want).abs().max() < 1e-5
    assert all(len(set(r)) == topk for r in idx.cpu().tolist())
    if copies >= topk:
        assert torch.equal(idx.long(), where[:topk].expand(nq, topk))
