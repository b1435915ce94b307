"""The candidate pools of the tensor-core sweep at the edges of their buffers and splits: kNN sets
against the FP64 oracle (certified ties allowed, no other difference)."""
import numpy as np
import pytest
import torch

import workloads
from tests import parity

pytestmark = pytest.mark.gpu


def _check(X, k, precision, pool=0, cam=None):
    import paper_2306_08792_gb300 as gcr
    X0 = gcr.gcr_normalize(torch.from_numpy(np.ascontiguousarray(X, dtype=np.float32)).cuda())
    n = X0.shape[0]
    p = gcr.default_params(k=k, precision=precision, pool=pool, cross_camera=0 if cam is None else 1, alpha=0.5)
    G = gcr.gcr_build_graph(X0, p, None if cam is None else torch.from_numpy(cam.astype(np.int32)).cuda())
    torch.cuda.synchronize()
    X64 = X0.double().cpu().numpy()
    r = parity.compare_knn(X64, np.arange(n), G.nbr.cpu().numpy(), k)
    assert r["mismatched"] == 0, r
    if cam is not None:
        rc = parity.compare_knn(X64, np.arange(n), G.nbr_cr.cpu().numpy(), k, cam, cross=True)
        assert rc["mismatched"] == 0, rc
    assert G.stats_dict()["band_failed"] == 0


# one tile and a column more, odd row blocks, splits of one and of several column tiles; pools of
# 32 (long rows take the deep ring), 64 and 128 entries, one and two graphs
@pytest.mark.parametrize("precision,n,d,k,pool,cams", [
    ("tf32", 257, 64, 10, 32, 0), ("tf32", 257, 64, 31, 32, 5), ("tf32", 2305, 1024, 20, 0, 0),
    ("tf32", 1537, 72, 40, 64, 0), ("tf32", 1537, 72, 40, 64, 4), ("bf16", 2817, 136, 15, 0, 6),
    ("tf32", 1100, 40, 60, 128, 0), ("tf32", 1100, 40, 60, 128, 3), ("tf32", 5000, 256, 12, 0, 0)])
def test_pool_sizes_and_splits(precision, n, d, k, pool, cams):
    X, cam = workloads.random_unit_like(n + d, n, d, cams=max(cams, 1))
    _check(X, k, precision, pool, cam if cams else None)


@pytest.mark.parametrize("precision,k,pool", [("tf32", 12, 32), ("tf32", 30, 64), ("tf32", 50, 128), ("bf16", 20, 64)])
def test_more_equal_scores_than_a_buffer_holds(precision, k, pool):
    """200 copies of one row and 40 of another among 1,500: every score a copy gives is tied
    far beyond the pool and its buffer."""
    rng = np.random.default_rng(4)
    X = rng.standard_normal((1500, 48)).astype(np.float32)
    X[rng.choice(1500, 200, replace=False)] = X[0]
    X[rng.choice(np.arange(1, 1500), 40, replace=False)] = X[1]
    _check(X, k, precision, pool)


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_scores_that_rise_or_fall_along_the_columns(sign):
    """Rows along an arc: for the last (first) rows every column tile beats all before it, so
    that every score is appended once and the buffers are compacted as often as they can be."""
    rng = np.random.default_rng(6)
    n, d = 1800, 64
    th = sign * np.linspace(0.0, 1.5, n)
    X = 0.04 * rng.standard_normal((n, d))
    X[:, 0] += np.cos(th)
    X[:, 1] += np.sin(th)
    _check(X, 20, "tf32")


# FP32 sweep: one tile and a column more, ragged splits, 32-, 64- and 128-entry pools of one and
# two graphs (two graphs of 128 entries take a sweep each), more ties than a buffer holds
@pytest.mark.parametrize("n,d,k,pool,cams", [
    (129, 20, 10, 32, 0), (257, 68, 31, 32, 5), (1537, 76, 40, 64, 0), (1537, 76, 40, 64, 4), (1100, 44, 60, 128, 0),
    (1100, 44, 60, 128, 3), (5000, 260, 15, 0, 0)])
def test_fp32_pool_sizes_and_splits(n, d, k, pool, cams):
    X, cam = workloads.random_unit_like(n + d, n, d, cams=max(cams, 1))
    _check(X, k, "fp32", pool, cam if cams else None)


@pytest.mark.parametrize("k,pool", [(12, 32), (30, 64)])
def test_fp32_equal_scores_go_to_the_smallest_columns(k, pool):
    """600 copies of one row: no pool can certify its rows, and the ones kept are the exact
    search's (ties to the smaller index)."""
    import paper_2306_08792_gb300 as gcr
    rng = np.random.default_rng(4)
    X = rng.standard_normal((1500, 48)).astype(np.float32)
    same = np.sort(rng.choice(np.arange(1, 1500), 600, replace=False))
    X[same] = X[0]
    same = np.concatenate([[0], same])
    X0 = gcr.gcr_normalize(torch.from_numpy(X).cuda())
    G = gcr.gcr_build_graph(X0, gcr.default_params(k=k, precision="fp32", pool=pool))
    nbr = np.sort(G.nbr.cpu().numpy()[same], axis=1)
    for t, i in enumerate(same):
        assert np.array_equal(nbr[t], same[same != i][:k]), (t, nbr[t])


@pytest.mark.parametrize("K,d", [(20, 64), (20, 520), (60, 64), (100, 64)])
def test_sampled_floors_of_a_wide_search(K, d):
    """300 queries against 60,001 rows: few row blocks and long splits, so a sample sweep gives the
    rows their floors (32- (both rings), 64- and 128-entry pools). A block of near-copies of some
    queries sits where the evenly spaced sample steps over it."""
    import paper_2306_08792_gb300 as gcr
    g = torch.Generator(device="cuda").manual_seed(K + d)
    G = torch.randn(60001, d, generator=g, device="cuda")
    Q = torch.randn(300, d, generator=g, device="cuda")
    G[1:59000:59][:200] = Q[:200] + 0.1 * torch.randn(200, d, generator=g, device="cuda")
    G, Q = gcr.gcr_normalize(G), gcr.gcr_normalize(Q)
    idx, dist = gcr.gcr_rerank(Q, G, gcr.default_params(precision="tf32", topk_out=K))
    ref = torch.cdist(Q.double(), G.double()).square()
    v, o = torch.topk(ref, K + 1, dim=1, largest=False)
    assert torch.allclose(dist.double(), v[:, :K], atol=2e-6, rtol=0)
    clear = v[:, K] - v[:, K - 1] > 1e-9
    assert torch.equal(idx[clear].long().sort(1)[0], o[clear, :K].sort(1)[0])


@pytest.mark.parametrize("ng", [1, 33, 64, 65, 256, 257, 511, 513, 1024, 1025, 2049])
def test_ranking_of_short_galleries(ng):
    """The bitonic network (to 256 keys) and the radix sort's small sizes, with exact ties."""
    import paper_2306_08792_gb300 as gcr
    rng = np.random.default_rng(ng)
    G = rng.standard_normal((ng, 40)).astype(np.float32)
    G[rng.choice(ng, ng // 4, replace=False)] = G[0]
    Q = rng.standard_normal((5, 40)).astype(np.float32)
    Xq, Xg = (gcr.gcr_normalize(torch.from_numpy(a).cuda()) for a in (Q, G))
    idx, dist = (t.cpu().numpy() for t in gcr.gcr_rerank(Xq, Xg, gcr.default_params(topk_out=0)))
    assert np.array_equal(np.sort(idx, axis=1), np.broadcast_to(np.arange(ng), idx.shape))
    step = np.diff(dist, axis=1)
    assert np.all(step >= 0) and np.all(np.diff(idx, axis=1)[step == 0] > 0)
    D = torch.cdist(Xq.double(), Xg.double()).square().cpu().numpy()
    # FP32 products of 40 terms: 40 * 2^-24, and the rounding of the distance
    assert np.max(np.abs(np.take_along_axis(D, idx, axis=1) - dist)) < 2 * 40 * 2.0 ** -24 + 3 * 2.0 ** -23


@pytest.mark.parametrize("precision", ["tf32", "bf16", "fp32"])
@pytest.mark.parametrize("K", [10, 100])
def test_wide_search_of_rows_that_meet_few_others(precision, K):
    """Queries of which five gallery rows, or none, have a positive score: the sampled floor is zero, and
    the rest of the list is the smallest indices among the rows of score zero (norms are exactly 1)."""
    import paper_2306_08792_gb300 as gcr
    ng = 300001
    G = torch.zeros(ng, 64, device="cuda")
    G[torch.arange(ng, device="cuda"), torch.arange(ng, device="cuda") % 32] = 1
    near = torch.tensor([7, 50000, 123456, 250001, ng - 1], device="cuda")
    G[near] = 0
    G[near, 40] = 1
    Q = torch.zeros(40, 64, device="cuda")
    Q[1::2, 40] = 1  # the even ones are zero rows
    idx, dist = gcr.gcr_rerank(Q, G, gcr.default_params(precision=precision, topk_out=K))
    idx = idx.long().cpu()
    all_rows = torch.arange(ng)
    others = all_rows[~torch.isin(all_rows, near.cpu())]
    assert torch.equal(idx[::2], all_rows[:K].expand(20, K))
    assert torch.equal(idx[1::2], torch.cat([near.cpu(), others[:K - 5]]).expand(20, K))
    assert torch.equal(dist[::2], torch.ones(20, K, device="cuda"))


@pytest.mark.parametrize("precision", ["fp32", "tf32", "bf16"])
@pytest.mark.parametrize("k,pool", [(15, 0), (40, 64)])
def test_rows_without_a_positive_score_take_the_smallest_columns(precision, k, pool):
    """900 of 3,000 unit rows are orthogonal to all others: every score of theirs is zero, every
    distance 2, and the ties go to the smaller index."""
    import paper_2306_08792_gb300 as gcr
    n = 3000
    alone = np.sort(np.random.default_rng(8).choice(n, 900, replace=False))
    col = np.arange(n) % 60
    col[alone] = 60 + np.arange(900)
    X = np.zeros((n, 960), dtype=np.float32)
    X[np.arange(n), col] = 1
    G = gcr.gcr_build_graph(torch.from_numpy(X).cuda(), gcr.default_params(k=k, precision=precision, pool=pool))
    nbr = np.sort(G.nbr.cpu().numpy()[alone], axis=1)
    first = np.arange(k + 1)
    for t, i in enumerate(alone):
        assert np.array_equal(nbr[t], first[first != i][:k]), (t, nbr[t])
