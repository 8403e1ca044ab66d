"""The norms of the 3-D multigrid's first pass count every cell once, in blocks of several tiles (few
planes) and of one (16 planes and more): ||alpha I0 + L_xy I0|| in 64 bits, from FP32-formed terms
(2^-22 relative)."""
import numpy as np
import pytest
import torch

from oracle import emfuse_oracle as O
from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 8, 32), (1, 9, 33), (1, 130, 1029), (2, 70, 300), (3, 65, 400), (5, 17, 700),
                                   (9, 33, 65), (15, 17, 70), (16, 17, 70), (17, 17, 70), (33, 9, 33)])
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
def test_right_hand_side_norm(shape, dtype):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    dev = torch.device("cuda", 0)
    I0 = torch.from_numpy(np.random.default_rng(71).integers(0, 256, size=shape)).to(dtype)
    _, st = api.emfuse_smooth_gradient_domain_mg(I0.to(dev), 0.25, return_stats=True)
    x = I0.double().numpy()
    assert st["b_norm"] == pytest.approx(float(np.linalg.norm(0.25 * x + O.laplacian(x))), rel=2.0 ** -22)
    assert st["converged"]
