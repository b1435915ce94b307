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


# few queries against so many rows that their norms take most of the array: fewer splits fit
@pytest.mark.parametrize("precision,nq,ng,d,topk", [
    ("fp32", 34, 577049, 664, 10), ("fp32", 91, 328194, 2552, 1), ("fp32", 11, 791863, 8, 63),
    ("fp32", 174, 376326, 616, 20), ("fp32", 63, 563776, 672, 10), ("fp32", 99, 423426, 2120, 10)])
def test_few_queries_against_many_rows_fit_the_static_scratch(precision, nq, ng, d, topk):
    import paper_2306_08792_gb300 as gcr
    from paper_2306_08792_gb300 import _lib
    p = gcr.default_params(precision=precision, topk_out=topk)
    need = _lib.load().gcr_rerank_workspace_size(nq, ng, d, ctypes.byref(p))
    assert 0 < need <= 16 << 20
