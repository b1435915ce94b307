"""Top-K re-rankings that fit the scratch of gcr_rerank_noalloc go on fitting it: the split buffers of
the FP32 sweep are the largest part for few queries against many rows."""
import ctypes

import pytest


@pytest.mark.parametrize("nq,ng,d,topk", [(100, 30000, 128, 10), (128, 30000, 1024, 20), (128, 60000, 1024, 10),
                                          (300, 8000, 1024, 20), (300, 16384, 1024, 10), (300, 60000, 1024, 20),
                                          (100, 16384, 128, 127)])
def test_few_queries_fit_the_static_scratch(nq, ng, d, topk):
    import paper_2306_08792_gb300 as gcr
    from paper_2306_08792_gb300 import _lib
    p = gcr.default_params(precision="fp32", topk_out=topk)
    need = _lib.load().gcr_rerank_workspace_size(nq, ng, d, ctypes.byref(p))
    assert 0 < need <= 16 << 20
