"""The direct solver over the whole range of alpha that its type holds: the gain alpha / (alpha +
lambda) stays in range where alpha times a coefficient does not.  s - o has a mean, which passes
with gain 1 at every alpha.  The bar is that of FP32 rounding through the transforms (100 half-ulps
of 512)."""
import numpy as np
import pytest
import torch

from oracle import emfuse_oracle as O
from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alpha", [1e-38, 1e-36, 1e-30, 1e-9, 1.0, 1e9, 1e30, 1e36, 3e38])
@pytest.mark.parametrize("precision", [api.PREC_FP32, api.PREC_FP64])
@pytest.mark.parametrize("shape", [(2, 301, 400), (1, 1, 1), (3, 1, 50)])
def test_extreme_alpha(alpha, precision, shape):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(31)
    o = rng.uniform(0, 200, size=shape).astype(np.float32)
    s = (o + 40 + rng.normal(0, 10, size=shape)).astype(np.float32)
    ref = np.stack([O.solve_dct(s[j], o[j], alpha) for j in range(shape[0])])
    f = api.emfuse_screened_poisson_dct(torch.from_numpy(s).to(dev), torch.from_numpy(o).to(dev), alpha, precision)
    assert np.max(np.abs(f.cpu().double().numpy() - ref)) <= 100 * 2.0 ** -24 * 512
