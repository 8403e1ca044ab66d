"""The 3-D multigrid below alpha = 1e-5 keeps its correction in FP64 at every tolerance: after the same
V-cycles, a call at tol 1e-7 (two floats at larger alpha) gives the bits of one at a tolerance that
asks for FP64, and conserves the mean as that one does."""
import numpy as np
import pytest
import torch

from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alpha", [1e-8, 1e-6, 9e-6])
@pytest.mark.parametrize("shape", [(24, 100, 101), (5, 64, 64)])
def test_correction_in_fp64(alpha, shape):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    dev = torch.device("cuda", 0)
    I0 = torch.from_numpy(np.random.default_rng(61).uniform(0, 255, size=shape).astype(np.float32)).to(dev)
    f, st = [None, None], [None, None]
    for q, tol in enumerate((1e-7, 1e-12)):
        f[q], st[q] = api.emfuse_smooth_gradient_domain_mg(I0, alpha, api.default_opts(tol=tol, max_vcycles=3),
                                                           return_stats=True, allow_noconv=True)
    assert st[0]["vcycles"] == st[1]["vcycles"] == 3
    assert torch.equal(f[0], f[1])
