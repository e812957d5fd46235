"""Feature statistics of the preconditioner network at the edges of binary32:
the sum of g^2 / d is formed in binary32 pairs where square and quotient fit,
and in FP64 where they do not."""
import numpy as np
import pytest

from gpu_common import cuda_tensor, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g,d", [(3.2e4, 2e-30), (1e14, 1e-29), (1e3, 2e-30), (1e16, 1e3), (1e-14, 1e25),
                                 (2e15, 1e34), (1e-20, 1e-25), (1.0, 3e38)])
def test_gradient_features_of_extreme_entries(g, d):
    """Every gradient feature is g / (sqrt(d) sum g^2 / d) clipped to [-4, 4],
    the sum in FP64 and rounded to binary32, to the rounding of BF16 (2^-8)."""
    import torch
    from paper_2112_05598_gb300 import LPC
    rng = np.random.default_rng(5)
    G, V = 8, 512
    diag = np.exp(rng.normal(size=(V, 4))).astype(np.float32)
    grad = (rng.normal(size=(V, 4)) * np.sqrt(diag) * 0.02).astype(np.float32)
    diag[77, 2], grad[77, 2] = d, g
    x, cross = rng.uniform(size=(V, 4)).astype(np.float32), np.zeros((V, 4), np.float32)
    feat = torch.empty(V, 16, dtype=torch.bfloat16, device="cuda")
    LPC(seed=1).features(G, cuda_tensor(x), cuda_tensor(grad), cuda_tensor(diag), cuda_tensor(cross), feat)
    d64, g64 = diag.astype(np.float64), grad.astype(np.float64)
    with np.errstate(over="ignore"):
        scale = np.float64(np.float32((g64 * g64 / d64).sum()))
    want = np.clip(g64 / (np.sqrt(d64) * scale), -4, 4)
    got = host(feat.float()).reshape(V, 16)[:, 7:11]
    assert np.all(np.isfinite(got))
    assert np.all(np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 1e-30)
