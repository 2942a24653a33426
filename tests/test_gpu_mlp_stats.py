"""Feature and target statistics of the learned target's training set, at sizes around the
kernel's split of the rows over the blocks of a cluster."""
import numpy as np
import pytest
import torch

from paper_2609_32920_gb300 import lt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 31, 255, 256, 511, 512, 513, 4095, 4096, 4097, 70001])
def test_statistics_match_float64(n):
    rng = np.random.default_rng(n)
    X = (rng.normal(size=(n, 16)) * rng.uniform(0.1, 3.0, 16) + rng.normal(size=16) * 5).astype(np.float32)
    T = (rng.normal(size=n) * 2 - 9).astype(np.float32)
    P = torch.zeros(lt.MLP_PARAMS, device="cuda")
    lt.mlp_init_stats(P, torch.tensor(X, device="cuda"), torch.tensor(T, device="cuda"))
    p = P.cpu().numpy().astype(np.float64)
    Xd, Td = X.astype(np.float64), T.astype(np.float64)
    # FP64 sums rounded to FP32 once; the variance loses mean^2 / var <= 1e4 of FP64's precision
    assert np.allclose(p[5313:5329], Xd.mean(0), rtol=1.2e-7, atol=1e-9)
    assert np.allclose(p[5329:5345], 1.0 / Xd.std(0), rtol=1.3e-7)
    assert np.allclose(p[5346], Td.mean(), rtol=1.2e-7)
    assert np.allclose(p[5345], Td.std(), rtol=1.3e-7)
    assert (p[:5313] == 0).all() and (p[5347:] == 0).all()
