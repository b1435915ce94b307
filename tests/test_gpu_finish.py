"""The block-wide selection that ends a search of many splits: one block's worth of entries, several
groups of splits, and more equal scores than it keeps."""
import ctypes

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


class _Gate(ctypes.Structure):
    _fields_ = [("flag", ctypes.c_void_p), ("want", ctypes.c_int)]


@pytest.mark.parametrize("S", [3, 12])
@pytest.mark.parametrize("kp,cap", [(32, 96), (128, 160)])
def test_counts_are_held_to_the_buffers(S, kp, cap):
    """Counts below zero or above the buffers' slots (a sweep that gave up a wait) are read as none
    and as all of them; the pools are the best of what the buffers then hold."""
    from paper_2306_08792_gb300 import _lib
    fn = _lib.load()["_ZN3gcr18launch_pool_finishEPKfPKiS3_iiiiiPfPiiiP11CUstream_stNS_4GateE"]
    fn.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int] * 5 + [ctypes.c_void_p] * 2 + [ctypes.c_int] * 2 + [
        ctypes.c_void_p, _Gate]
    rng = np.random.default_rng(S + kp)
    kinds, rows = 2, 5
    v = rng.standard_normal((S, kinds * rows, cap)).astype(np.float32)
    i = (np.arange(S)[:, None, None] * 1000 + rng.permuted(np.tile(np.arange(cap), (S, kinds * rows, 1)), axis=2))
    cnt = rng.choice([-2**31, -1, 0, 1, kp, cap, cap + 1, 2**31 - 1], size=(S, kinds * rows))
    dv, di, dc = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (v, i.astype(np.int32), cnt.astype(np.int32)))
    ov = torch.empty(kinds * rows, kp, device="cuda")
    oi = torch.empty(kinds * rows, kp, dtype=torch.int32, device="cuda")
    assert fn(dv.data_ptr(), di.data_ptr(), dc.data_ptr(), S, kinds, rows, cap, kp, ov.data_ptr(), oi.data_ptr(), rows,
              0, torch.cuda.current_stream().cuda_stream, _Gate(None, 0)) == 0
    for w in range(kinds * rows):
        keep = [(-v[s, w, e], i[s, w, e]) for s in range(S) for e in range(min(max(int(cnt[s, w]), 0), cap))]
        want = sorted(keep)[:kp]
        got = oi[w].cpu().numpy()
        assert np.array_equal(got[:len(want)], [c for _, c in want]) and np.all(got[len(want):] == -1)
        assert np.array_equal(ov[w].cpu().numpy()[:len(want)], [-x for x, _ in want])
