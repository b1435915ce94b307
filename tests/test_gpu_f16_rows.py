"""Serving in TF32 mode on unit rows at the ends of the range of their 16-bit copies: elements of
1, and neighbours told apart only by elements that lose bits in the copy (below 2^-28) or vanish
in it (below 2^-39)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,hi", [(2.0 ** -31, 2.0 ** -29), (2.0 ** -41, 2.0 ** -39)])
def test_neighbours_told_apart_below_the_copies_range(lo, hi):
    """24 rows of 3,000 are a unit vector plus such elements: the copies give them equal scores but
    for bits far below the rounding bound. The ten nearest of each query are the FP64 ranking's: the
    boundary is settled by FP64 dot products, whose terms of 64 elements round six times by at most
    2^-53 (1e-15 with the norms' part; the tenth and eleventh lie further apart)."""
    import paper_2306_08792_gb300 as gcr
    from paper_2306_08792_gb300.serving import Gallery
    g = torch.Generator().manual_seed(11)
    X = torch.randn(3000, 64, generator=g)
    near = torch.randperm(3000, generator=g)[:24]
    t = (lo + (hi - lo) * torch.rand(24, 32, generator=g)) * torch.where(torch.rand(24, 32, generator=g) < 0.5, -1.0, 1.0)
    X[near] = 0.0
    X[near, 0] = 1.0
    X[near[:, None], torch.arange(32, 64)[None]] = t
    Q = torch.zeros(5, 64)
    Q[:, 0] = 1.0
    Q[:, 32:] = 0.125 * torch.where(torch.rand(5, 32, generator=g) < 0.5, -1.0, 1.0)
    p = gcr.default_params(k=5, T=0, precision="tf32", topk_out=10)
    Xg, Xq = gcr.gcr_normalize(X.cuda()), gcr.gcr_normalize(Q.cuda())
    assert torch.equal(Xg[near].cpu(), X[near])  # unit rows already
    s = Xq.double().cpu()[:, 32:] @ Xg.double().cpu()[near][:, 32:].T  # (the rest of the scores is common)
    v, o = s.sort(dim=1, descending=True)
    idx, dist = Gallery(X.cuda(), p).query(Q.cuda())
    torch.cuda.synchronize()
    idx = idx.cpu().long()
    assert torch.isin(idx, near).all() and torch.isfinite(dist).all()
    for q in range(5):
        assert v[q, 9] - v[q, 10] > 1e-15
        assert set(idx[q].tolist()) == set(near[o[q, :10]].tolist())
