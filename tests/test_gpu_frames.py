"""The frame passes of the profile vectors at the edges of their batches (8 frames) and column
slices (512 and 1,024 floats)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

LENGTHS = [1, 15, 16, 17, 2, 33, 1, 5, 31, 32]


def _frames(d):
    rng = np.random.default_rng(d)
    off = np.concatenate([[0], np.cumsum(LENGTHS)]).astype(np.int64)
    F = rng.standard_normal((len(LENGTHS), d)).repeat(LENGTHS, axis=0) + 0.7 * rng.standard_normal((off[-1], d))
    return F.astype(np.float32), off


@pytest.mark.parametrize("d", [4, 512, 516, 1024, 1028, 2048, 2052, 4096])
def test_profiles_and_means(d):
    """The bounds of tests/test_gpu_gcrv.py: means 1e-6, profiles 2e-5 after normalisation (Gram operands
    of 2^-16, divided by lambda = 10; conjugate gradients to 1e-7)."""
    import paper_2306_08792_gb300 as gcr
    F, off = _frames(d)
    cam = np.array([0, 1] * 5, np.int32)
    Fd, od = torch.from_numpy(F).cuda(), torch.from_numpy(off).cuda()
    mu = gcr.gcrv_mean_profiles(Fd, od).double().cpu().numpy()
    np.testing.assert_allclose(mu, oracle.mean_profiles(oracle.l2_normalize(F), off), atol=1e-6, rtol=0)
    W = gcr.gcrv_profiles(Fd, od, torch.from_numpy(cam).cuda(), 2, 10.0).double().cpu().numpy()
    Wo = oracle.pvg_profiles(F, off, cam, 10.0)
    nW, nWo = np.linalg.norm(W, axis=1, keepdims=True), np.linalg.norm(Wo, axis=1, keepdims=True)
    np.testing.assert_allclose(W / nW, Wo / nWo, atol=2e-5, rtol=0)
    np.testing.assert_allclose(nW, nWo, rtol=1e-4)


@pytest.mark.parametrize("C,d", [(303, 68), (304, 68), (7, 1024), (5, 1636), (4, 2044), (2, 4092), (1, 4096), (2, 4096)])
def test_means_of_few_long_and_of_many_tracklets(C, d):
    """Both forms of the frame pass (norms first, or with the means) at the line between them, ragged."""
    import paper_2306_08792_gb300 as gcr
    rng = np.random.default_rng(C + d)
    length = rng.integers(1, 60, size=C)
    off = np.concatenate([[0], np.cumsum(length)]).astype(np.int64)
    F = rng.standard_normal((off[-1], d)).astype(np.float32)
    mu = gcr.gcrv_mean_profiles(torch.from_numpy(F).cuda(), torch.from_numpy(off).cuda()).double().cpu().numpy()
    np.testing.assert_allclose(mu, oracle.mean_profiles(oracle.l2_normalize(F), off), atol=1e-6, rtol=0)
