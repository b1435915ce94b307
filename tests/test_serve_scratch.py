"""A workspace sized for a batch of queries serves every smaller batch (the serving loop's slots hold
one of the largest batch): the size never falls as the batch grows. Host queries only."""
import ctypes

import numpy as np
import pytest


def _sizes(precision, ng, d, k, topk, batches):
    import paper_2306_08792_gb300 as gcr
    from paper_2306_08792_gb300 import _lib
    p = gcr.default_params(precision=precision, k=k, T=2, topk_out=topk)
    lib = _lib.load()
    return np.array([lib.gcr_serve_workspace_size(b, ng, d, ctypes.byref(p)) for b in batches], dtype=np.int64)


@pytest.mark.parametrize("ng,d,k,topk", [(50021, 256, 20, 100), (14601, 1024, 5, 100), (102437, 128, 30, 100),
                                         (20000, 256, 20, 20), (500000, 256, 20, 100)])
@pytest.mark.parametrize("precision", ["fp32", "tf32", "bf16"])
def test_no_batch_needs_more_than_a_larger_one(precision, ng, d, k, topk):
    s = _sizes(precision, ng, d, k, topk, range(1, 641))
    assert s[0] > 0 and np.all(np.diff(s) >= 0)


@pytest.mark.parametrize("precision", ["fp32", "tf32", "bf16"])
def test_random_galleries(precision):
    rng = np.random.default_rng(11)
    for _ in range(60):
        ng = int(np.exp(rng.uniform(np.log(2000), np.log(2e6))))
        d = 8 * int(np.exp(rng.uniform(0, np.log(128))))
        s = _sizes(precision, ng, d, int(rng.choice([5, 20, 50])), int(rng.choice([5, 31, 50, 127])),
                   [*range(1, 520, 9), 1023, 2048])
        assert s[0] > 0 and np.all(np.diff(s) >= 0), (ng, d)
