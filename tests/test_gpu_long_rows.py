"""Smoothing along a very long axis: normalisers formed once for the inner cells and one by one at the
two ends, on x, y and z, beside axes shorter than the support, against the oracle.  A pass
of n taps errs by at most (n + 3) 2^-24 255, and a following pass does not enlarge it."""
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


@pytest.mark.parametrize("shape", [(2, 3, 20001), (2, 3, 20016), (1, 20001, 2), (3000, 2, 3), (1, 1, 20011)])
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
@pytest.mark.parametrize("sigmas", [(1.0, 3.0), (0.5, 0.5), (4.0, 5.0)])
def test_long_axis(dev, shape, dtype, sigmas):
    I0 = torch.from_numpy(np.random.default_rng(51).integers(0, 256, size=shape)).to(dtype)
    out = api.emfuse_smooth_z(I0.to(dev), *sigmas).cpu().double().numpy()
    ref = O.smooth_stack(I0.double().numpy(), *sigmas)
    taps = [2 * O.support_radius(s) + 1 for s in sigmas]
    assert np.abs(out - ref).max() <= (2 * (taps[0] + 3) + taps[1] + 3) * 2.0 ** -24 * 255.0
