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
