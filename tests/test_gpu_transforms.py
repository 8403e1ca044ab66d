"""The cosine transforms of the direct solvers at the sizes where their index arithmetic has
cases of its own: sides of 1 (one-dimensional and trivial transforms), even and odd lengths (a
mode that is its own mirror image or not), and both at once."""
import numpy as np
import pytest
import torch

from oracle import emfuse_oracle as O
from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu

SHAPES = [(3, 1, 1), (1, 1, 2), (2, 2, 1), (2, 1, 9), (1, 9, 1), (2, 2, 2), (1, 3, 2), (2, 2, 3), (1, 3, 3), (3, 4, 5),
          (1, 37, 64), (2, 64, 37), (1, 257, 258)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch.device("cuda", 0)


def close(f, ref, precision):
    """FP64 transforms: the rounding of the FP32 output (half an ulp below 512, 1.6e-5) with as
    much again for the transforms.  FP32: 24-bit rounding through about 2 log2(n) + nz stages of
    values up to 512, less than 100 half-ulps."""
    bar = 3.2e-5 if precision == api.PREC_FP64 else 100 * 2.0 ** -24 * 512
    assert np.max(np.abs(f.cpu().double().numpy() - ref)) <= bar


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision", [api.PREC_FP32, api.PREC_FP64])
def test_slice_solve(dev, shape, precision):
    rng = np.random.default_rng(11)
    s = rng.uniform(0, 255, size=shape).astype(np.float32)
    o = np.clip(0.9 * s + rng.normal(0, 10, size=shape), 0, 255).astype(np.float32)
    ref = np.stack([O.solve_dct(s[j], o[j], 0.01) for j in range(shape[0])])
    f = api.emfuse_screened_poisson_dct(torch.from_numpy(s).to(dev), torch.from_numpy(o).to(dev), 0.01, precision)
    close(f, ref, precision)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dtype", [torch.float32, torch.uint8])
@pytest.mark.parametrize("precision", [api.PREC_FP32, api.PREC_FP64])
def test_gradient_domain(dev, shape, dtype, precision):
    I0 = torch.from_numpy(np.random.default_rng(12).integers(0, 256, size=shape)).to(dtype)
    ref = O.gradient_domain_smooth(I0.double().numpy(), 0.05)
    close(api.emfuse_smooth_gradient_domain(I0.to(dev), 0.05, precision), ref, precision)
