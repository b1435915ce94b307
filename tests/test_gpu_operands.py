"""The 16-bit operands of TF32 mode: the first layer of a large problem is searched on FP16 copies
that hold the TF32-rounded values, and again on TF32 where the ball search would run."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("noise,ball", [(0.3, False), (0.002, True)])
@pytest.mark.parametrize("k", [20, 30])
def test_first_layer_search_equals_the_tf32_search(noise, ball, k):
    """20,000 rows of d = 512 in clusters of about 100. Local propagation searches its normalised
    input as a first layer; gcr_build_graph takes any rows and stays on TF32. The lists are the same,
    and so are the counters where the search was repeated (noise 0.002: contracted clusters)."""
    import paper_2306_08792_gb300 as gcr
    g = torch.Generator(device="cuda").manual_seed(3)
    cent = torch.randn(200, 512, generator=g, device="cuda")
    lab = torch.randint(0, 200, (20000,), generator=g, device="cuda")
    X = cent[lab] + noise * torch.randn(20000, 512, generator=g, device="cuda")
    p = gcr.default_params(k=k, T=1, precision="tf32")
    ds = gcr.Dsfp(20000, 512, p)
    ds(X)
    G = gcr.gcr_build_graph(gcr.gcr_normalize(X), p)
    assert torch.equal(ds.nbr[:, :k], G.nbr)
    st = G.stats_dict()
    assert (st["ball_groups"] > 0) == ball and st["band_failed"] == 0, st
    if ball:
        assert ds.stats.cpu().tolist() == G.stats.cpu().tolist()


def test_scaled_fp16_holds_the_tf32_rounded_value():
    """Rounding to 11 significant bits, then times 2^14: the conversion to FP16 is exact for every
    element of a unit row down to 2^-28 (and off by at most 2^-39 below)."""
    x = np.concatenate([np.ldexp(np.random.default_rng(1).uniform(0.5, 1.0, 200), -e) for e in range(0, 40)])
    x = x.astype(np.float32)
    t = ((x.view(np.uint32) + 0x1000) & 0xFFFFE000).view(np.float32)
    back = (t * np.float32(16384.0)).astype(np.float16).astype(np.float64) / 16384.0
    big = x >= 2.0 ** -28
    assert np.array_equal(back[big], t[big].astype(np.float64))
    assert np.max(np.abs(back - t)) <= 2.0 ** -39


@pytest.mark.parametrize("noise", [0.3, 0.02])
def test_later_layers_equal_the_tf32_search(noise):
    """Two layers of 20,000 rows of d = 512, by gcr_pipeline (later layers are probed, and searched
    on 16-bit copies or on TF32) and layer by layer through gcr_build_graph (TF32): X_T and the
    ranking are the same bits."""
    import paper_2306_08792_gb300 as gcr
    g = torch.Generator(device="cuda").manual_seed(5)
    cent = torch.randn(400, 512, generator=g, device="cuda")
    lab = torch.randint(0, 400, (20000,), generator=g, device="cuda")
    X = cent[lab] + noise * torch.randn(20000, 512, generator=g, device="cuda")
    p = gcr.default_params(k=20, T=2, precision="tf32", topk_out=50)
    idx, dist, XT, st = gcr.gcr_pipeline(X, 500, p)
    Y = gcr.gcr_normalize(X)
    for _ in range(2):
        Y = gcr.gcr_propagate(gcr.gcr_build_graph(Y, p), Y)
    assert torch.equal(XT, Y)
    i2, d2 = gcr.gcr_rerank(Y[:500].contiguous(), Y[500:].contiguous(), p)
    assert torch.equal(idx, i2) and torch.equal(dist, d2)
