"""The 3-D multigrid's passes (tiles of 64 x 64 columns marching along z in chunks, an odd number
of passes per leg, the small levels in one CTA) at the sizes and sweep counts where their index
arithmetic has cases of its own: tile edges, rows of odd length (unaligned pairs in the caller's
output buffer), partial cells on each axis, one plane, one column, chunks along z, and 0 to 4 sweeps
per leg.  The bar is the residual's own: ||f - f*|| <= ||r|| / alpha (A >= alpha I), with the FP32
output's rounding."""
import math

import numpy as np
import pytest
import torch

from oracle import emfuse_oracle as O
from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu

SHAPES = [(1, 53, 57), (2, 113, 104), (40, 60, 60), (3, 130, 229), (17, 1, 900), (9, 1000, 1), (33, 52, 53), (5, 64, 65)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch.device("cuda", 0)


def check(dev, shape, dtype, alpha, **kw):
    I0 = torch.from_numpy(np.random.default_rng(3).integers(0, 256, size=shape)).to(dtype)
    ref = O.gradient_domain_smooth(I0.double().numpy(), alpha)
    f, st = api.emfuse_smooth_gradient_domain_mg(I0.to(dev), alpha, api.default_opts(max_vcycles=80, **kw),
                                                 return_stats=True)
    assert st["converged"]
    err = float(np.linalg.norm(f.cpu().double().numpy() - ref))
    assert err <= 1.01 * st["rel_residual"] * st["b_norm"] / alpha + 512 * 2.0 ** -24 * math.sqrt(I0.numel())


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dtype", [torch.float32, torch.uint8])
@pytest.mark.parametrize("tol", [1e-6, 1e-8])  # the correction in two floats / in FP64
def test_sizes(dev, shape, dtype, tol):
    check(dev, shape, dtype, 0.1, tol=tol)


@pytest.mark.parametrize("nu", [(1, 1), (3, 2), (2, 3), (4, 1), (0, 2), (2, 0)])
@pytest.mark.parametrize("first", [1, 3])
def test_sweeps(dev, nu, first):
    check(dev, (12, 120, 71), torch.float32, 0.1, nu_pre=nu[0], nu_post=nu[1], first_vcycles=first)
