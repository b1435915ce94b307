"""Searches of more than 65,536 columns (splits that the 16-bit column offsets force) whose rows are
swept in chunks that share the splits' buffers."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _check_rows(X, rows, nbr, k, cam=None):
    """The k nearest of the given rows against FP64: every neighbour within 1e-9 of the k-th distance."""
    for r in rows.split(64):
        D = (X[r, None].double() - 0).square().sum(-1) + X.double().square().sum(-1) - 2 * X[r].double() @ X.double().T
        D[torch.arange(len(r), device="cuda"), r] = float("inf")
        if cam is not None:
            D[cam[r][:, None] == cam[None, :]] = float("inf")
        kth = D.topk(k, dim=1, largest=False).values[:, -1:]
        got = D.gather(1, nbr[r].long())
        assert (got <= kth + 1e-9).all()
        assert all(len(set(t)) == k for t in nbr[r].cpu().tolist())


@pytest.mark.parametrize("precision,k,cams", [("tf32", 15, 0), ("tf32", 25, 4), ("bf16", 15, 0), ("fp32", 15, 0),
                                              ("fp32", 15, 4)])
def test_graph_of_several_chunks_and_forced_splits(precision, k, cams):
    """180,001 rows: three splits by their columns, two chunks (three with both graphs). Rows around
    every multiple of 128 rows of the middle third, the splits' ends, the ragged last block, and
    a random sample."""
    import paper_2306_08792_gb300 as gcr
    n = 180001
    g = torch.Generator(device="cuda").manual_seed(21)
    X = gcr.gcr_normalize(torch.randn(n, 24, generator=g, device="cuda"))
    cam = torch.randint(0, cams, (n,), generator=g, device="cuda").int() if cams else None
    p = gcr.default_params(k=k, precision=precision, cross_camera=1 if cams else 0, alpha=0.5)
    G = gcr.gcr_build_graph(X, p, cam)
    torch.cuda.synchronize()
    edge = torch.arange(59904, 120192, 2048, device="cuda")
    rows = torch.cat([edge - 1, edge, torch.tensor([0, 127, 128, 65535, 65536, 131071, 131072, n - 2, n - 1], device="cuda"),
                      torch.randint(0, n, (150,), generator=g, device="cuda")])
    _check_rows(X, rows, G.nbr, k)
    if cams:
        _check_rows(X, rows, G.nbr_cr, k, cam)
    assert G.stats_dict()["band_failed"] == 0 and G.stats_dict()["saturated"] == 0


def test_search_of_several_chunks_with_sampled_floors():
    """3,100 queries of 4,700,003 rows, 100 best: 72 splits and more, each chunk with its own sample sweep.
    FP32 distances of 8 terms: within 1e-6 of FP64, and every index at its distance."""
    import paper_2306_08792_gb300 as gcr
    g = torch.Generator(device="cuda").manual_seed(22)
    G = gcr.gcr_normalize(torch.randn(4700003, 8, generator=g, device="cuda"))
    Q = gcr.gcr_normalize(torch.randn(3100, 8, generator=g, device="cuda"))
    idx, dist = gcr.gcr_rerank(Q, G, gcr.default_params(precision="tf32", topk_out=100))
    pick = torch.cat([torch.arange(0, 3100, 97), torch.tensor([1535, 1536, 1663, 1664, 3099])]).cuda()
    for r in pick.split(16):
        D = 2.0 - 2.0 * Q[r].double() @ G.double().T
        want = D.topk(100, dim=1, largest=False).values
        assert (D.gather(1, idx[r].long()) - want).abs().max() < 1e-6
        assert (dist[r].double() - want).abs().max() < 1e-6
