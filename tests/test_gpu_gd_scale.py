"""The 3-D gradient-domain multigrid is linear: input scaled by a power of two, up to where squares
leave the FP32 range (2^-80, 2^66), takes the same V-cycles to the scaled result.  Every operation
scales exactly but for underflow of low-order parts, so the bar is two ulps of the 8-bit range
(2^-15), and the norms, summed in FP64, agree to the same 2^-22."""
import numpy as np
import pytest
import torch

from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch.device("cuda", 0)


@pytest.mark.parametrize("exponent", [-80, -66, 40, 60, 66])
@pytest.mark.parametrize("tol", [1e-6, 1e-8])  # the correction in two floats / in FP64
def test_scaled_input(dev, exponent, tol):
    rng = np.random.default_rng(8)
    I0 = torch.from_numpy(rng.uniform(0, 255, size=(18, 70, 83)).astype(np.float32)).to(dev)
    opts = api.default_opts(tol=tol)
    f, st = api.emfuse_smooth_gradient_domain_mg(I0, 0.1, opts, return_stats=True)
    scale = 2.0 ** exponent
    g, sg = api.emfuse_smooth_gradient_domain_mg(I0 * scale, 0.1, opts, return_stats=True)
    assert sg["converged"] and sg["vcycles"] == st["vcycles"]
    assert sg["b_norm"] == pytest.approx(st["b_norm"] * scale, rel=2.0 ** -22)
    assert sg["rel_residual"] == pytest.approx(st["rel_residual"], rel=1e-2)
    assert float((g / scale - f).abs().max()) <= 2.0 ** -15
