"""The general smoothing passes and their adjoint on narrow stacks, whose rows are taken as one line of
cells, on either side of that rule's line (64 cells a row), and the z pass over planes taken as one
row.  Tolerances: a pass of n taps forms a weighted mean of values <= 255 with rounded taps and
normaliser, so it errs by at most (n + 3) 2^-24 255, and a following pass does not enlarge an earlier
one's error; the gradients carry the solve's error (relative residual 1e-6) besides: 1e-4 of their
largest value."""
import numpy as np
import pytest
import torch

from oracle import emfuse_oracle as O
from paper_1506_02079_gb300 import api
from paper_1506_02079_gb300.synthetic import make_stack

pytestmark = pytest.mark.gpu

SHAPES = [(7, 129, 3), (5, 40, 20), (9, 17, 63), (9, 17, 64), (3, 1, 47), (40, 2, 2), (2, 33, 1)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch.device("cuda", 0)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
@pytest.mark.parametrize("sigmas", [(3.0, 1.0), (1.0, 3.5), (10.5, 10.5)])
def test_general_smoothing(dev, shape, dtype, sigmas):
    I0 = make_stack(*shape, seed=12, out_dtype=dtype)
    out = api.emfuse_smooth_z(I0.to(dev), *sigmas).cpu().double().numpy()
    ref = O.smooth_stack(I0.double().numpy(), *sigmas)
    taps = [2 * O.support_radius(s) + 1 for s in sigmas]
    assert np.abs(out - ref).max() <= (2 * (taps[0] + 3) + taps[1] + 3) * 2.0 ** -24 * 255.0


@pytest.mark.parametrize("shape", SHAPES)
def test_adjoint(dev, shape):
    alpha, sigmas = 0.3, (1.0, 2.5)
    I0 = make_stack(*shape, seed=6)
    g = torch.from_numpy(np.random.default_rng(10).normal(size=shape)).float()
    Id = I0.to(dev)
    s = api.emfuse_smooth_z(Id, *sigmas)
    f = api.emfuse_screened_poisson(s, Id, alpha)
    got = api.emfuse_backward(g.to(dev), f, s, Id, *sigmas, alpha)
    x, gd = I0.double().numpy(), g.double().numpy()
    dI0, _, dsig = O.backward_stack(gd, x, *sigmas, alpha)
    lam = np.stack([O.apply_Ainv(gj, alpha) for gj in gd])
    assert np.abs(got["in0"].cpu().numpy() - dI0).max() <= 1e-4 * np.abs(dI0).max()
    assert abs(got["sigma_z"] - dsig) <= 1e-4 * np.abs(alpha * lam * O.dsmooth_dsigma_z(x, *sigmas)).sum()
