"""The serving loop's smaller batches in the workspace of its largest (FP32: fewer rows, more splits)."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


def test_fp32_buckets_in_the_workspace_of_the_largest():
    import paper_2306_08792_gb300 as gcr
    from paper_2306_08792_gb300.serving import Gallery, Server, make_requests
    w = workloads.serving(seed=7, n_gallery=14601, d=1024, n_clusters=700, n_requests=24, rate=2000.0, max_batch=64)
    p = gcr.default_params(k=5, T=2, topk_out=100, precision="fp32")
    G = Gallery(torch.from_numpy(w.gallery).cuda(), p)
    srv = Server(G, n_slots=2, max_batch=128)
    srv.warmup(sizes=(1, 2, 4, 8, 16, 32, 64, 128))
    reqs = make_requests(w, 24, realtime=False)
    assert srv.run(reqs, realtime=False)["requests"] == 24
    for r in reqs[::3]:
        i, d = G.query(torch.from_numpy(r.queries).cuda())
        assert np.array_equal(i.cpu().numpy(), r.idx)
        np.testing.assert_allclose(d.cpu().numpy(), r.dist, atol=1e-6, rtol=0)


@pytest.mark.parametrize("nq,ng,topk", [(34, 577049, 10), (11, 791863, 63)])
def test_top_k_in_the_static_scratch_with_fewer_splits(nq, ng, topk):
    """The distances of the K nearest, in order, within 1e-5 (FP32 dot products of 32 terms), and
    every index at its distance."""
    import paper_2306_08792_gb300 as gcr
    g = torch.Generator(device="cuda").manual_seed(nq)
    q = gcr.gcr_normalize(torch.randn(nq, 32, generator=g, device="cuda"))
    b = gcr.gcr_normalize(torch.randn(ng, 32, generator=g, device="cuda"))
    idx = torch.empty(nq, topk, dtype=torch.int32, device="cuda")
    dist = torch.empty(nq, topk, device="cuda")
    gcr.gcr_rerank_noalloc(q, b, gcr.default_params(precision="fp32", topk_out=topk), idx, dist)
    D = 2.0 - 2.0 * (q.double() @ b.double().T)
    want = D.topk(topk, dim=1, largest=False).values
    assert (D.gather(1, idx.long()) - want).abs().max() < 1e-5 and (dist.double() - want).abs().max() < 1e-5
    assert all(len(set(r)) == topk for r in idx.cpu().tolist())
