"""The scratch of a search is linear in its rows: the splits that the 16-bit column offsets force share
one region, chunk by chunk. Host queries only."""
import ctypes

import pytest


def _need(fn, n, d, **kw):
    import paper_2306_08792_gb300 as gcr
    from paper_2306_08792_gb300 import _lib
    p = gcr.default_params(**kw)
    return getattr(_lib.load(), fn)(n, d, ctypes.byref(p))


# bytes a row when every row keeps one list instead of a buffer per split (the version before these
# buffers); the two graphs at k = 30, pools of 64, take 15,200
@pytest.mark.parametrize("n,d,precision,k,cross,row", [
    (4_000_000, 64, "tf32", 20, 0, 7590), (4_000_000, 64, "tf32", 30, 1, 15180), (1_000_000, 128, "tf32", 20, 0, 9130),
    (2_000_000, 256, "fp32", 20, 0, 5040), (16_000_000, 64, "tf32", 20, 0, 7590)])
def test_graph_scratch_per_row_stays_bounded(n, d, precision, k, cross, row):
    need = _need("gcr_build_graph_workspace_size", n, d, precision=precision, k=k, cross_camera=cross)
    assert 0 < need <= 1.1 * row * n


@pytest.mark.parametrize("precision", ["fp32", "tf32", "bf16"])
@pytest.mark.parametrize("fn", ["gcr_build_graph_workspace_size", "gcr_gallery_build_workspace_size",
                                "gcr_dsfp_workspace_size"])
def test_scratch_is_linear_in_the_rows(fn, precision):
    kw = dict(precision=precision, k=20, T=2, topk_out=100)
    one = _need(fn, 1_000_000, 64, **kw)
    assert _need(fn, 8_000_000, 64, **kw) <= 8.1 * one
