"""The local propagation's register tiles at the edges of their ranges: the largest and smallest
numbers of local rows of each tile size (4, 6, 7 and 8 rows), the first past them, and column counts
below, at and past a chunk of 128."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

# As tests/test_gpu_dsfp.py: the Gram's FP32 dot products (~1e-6 at d = 4096) moved through
# exp(-d2 / gamma) by 1 / gamma = 5.
TOL = 5e-6


@pytest.mark.parametrize("k", [2, 4, 11, 12, 17, 18, 20, 21, 23, 24, 31, 32])
@pytest.mark.parametrize("d", [4, 128, 132, 520])
def test_tiles_match_oracle(k, d):
    import paper_2306_08792_gb300 as gcr
    n = 90
    rng = np.random.default_rng(100 * k + d)
    cent = rng.standard_normal((6, d))
    U32 = oracle.l2_normalize(cent[rng.integers(0, 6, n)] + 0.5 * rng.standard_normal((n, d))).astype(np.float32)
    U64 = U32.astype(np.float64)
    nbr = oracle.knn(U64, k)[0].astype(np.int32)
    nbr[3, k // 2:] = -1   # absent neighbours, also between present ones
    nbr[5, ::2] = -1
    nbr[7, :] = -1
    Y = gcr.gcr_dsfp_propagate(torch.from_numpy(U32).cuda(), torch.from_numpy(nbr).cuda(), 0.2, 2).cpu().numpy()
    ref = np.array([oracle.dsfp_local(U64, i, nbr[i], 0.2, 2) for i in range(n)])
    assert np.abs(Y - ref).max() < TOL
