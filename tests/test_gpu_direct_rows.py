"""The direct solvers' passes over few long rows, several blocks to a row, and over many short ones,
one block to several: lengths about the block's 256 threads and the multiples that one round of
blocks covers (152 x 32 blocks)."""
import numpy as np
import pytest
import torch

from oracle import emfuse_oracle as O
from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch.device("cuda", 0)


@pytest.mark.parametrize("shape", [(1, 2, 255), (1, 2, 257), (2, 3, 513), (1, 2, 70000), (1, 1, 150001), (1, 150001, 1),
                                   (4870, 1, 3), (2440, 2, 2)])
@pytest.mark.parametrize("precision", [api.PREC_FP32, api.PREC_FP64])
def test_row_passes(dev, shape, precision):
    rng = np.random.default_rng(41)
    s = rng.uniform(0, 255, size=shape).astype(np.float32)
    o = np.clip(0.9 * s + rng.normal(0, 10, size=shape), 0, 255).astype(np.float32)
    # the rounding of the FP32 output with as much again in FP64; 100 half-ulps of 512 in FP32
    bar = 3.2e-5 if precision == api.PREC_FP64 else 100 * 2.0 ** -24 * 512
    f = api.emfuse_screened_poisson_dct(torch.from_numpy(s).to(dev), torch.from_numpy(o).to(dev), 0.01, precision)
    ref = np.stack([O.solve_dct(s[j], o[j], 0.01) for j in range(shape[0])])
    assert np.max(np.abs(f.cpu().double().numpy() - ref)) <= bar
    if shape[0] < 100:
        g = api.emfuse_smooth_gradient_domain(torch.from_numpy(s).to(dev), 0.05, precision)
        assert np.max(np.abs(g.cpu().double().numpy() - O.gradient_domain_smooth(s.astype(np.float64), 0.05))) <= bar
