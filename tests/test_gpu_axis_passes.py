"""The general smoothing passes along x, y and z, their transposes and the adjoint's Laplacian at the
sizes where they can go wrong: rows around 32 and 128 cells, axes around groups of 8 cells, axes
shorter than the support, one cell.

Tolerances: a pass of n taps forms a weighted mean of values <= 255 with rounded taps and normaliser, so it
errs by at most (n + 3) 2^-24 255, and a following pass does not enlarge an earlier one's error.
The gradients carry the solve's error besides (relative residual 1e-6): 1e-4 of their largest
value, and of the sum of the absolute products for the scalar one."""
import numpy as np
import pytest
import torch

from oracle import emfuse_oracle as O
from paper_1506_02079_gb300 import api
from paper_1506_02079_gb300.synthetic import make_stack

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (2, 33, 31), (7, 8, 128), (9, 17, 129), (17, 9, 257), (24, 40, 33)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch.device("cuda", 0)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
@pytest.mark.parametrize("sigmas", [(3.0, 1.0), (1.0, 3.5), (10.5, 10.5)])
def test_general_smoothing(dev, shape, dtype, sigmas):
    I0 = make_stack(*shape, seed=11, out_dtype=dtype)
    out = api.emfuse_smooth_z(I0.to(dev), *sigmas).cpu().double().numpy()
    ref = O.smooth_stack(I0.double().numpy(), *sigmas)
    taps = [2 * O.support_radius(s) + 1 for s in sigmas]
    assert np.abs(out - ref).max() <= (2 * (taps[0] + 3) + taps[1] + 3) * 2.0 ** -24 * 255.0


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("sigmas", [(1.0, 2.5), (3.0, 0.5), (0.0, 4.0)])
def test_adjoint(dev, shape, sigmas):
    alpha = 0.3
    I0 = make_stack(*shape, seed=5)
    g = torch.from_numpy(np.random.default_rng(9).normal(size=shape)).float()
    Id = I0.to(dev)
    s = api.emfuse_smooth_z(Id, *sigmas)
    f = api.emfuse_screened_poisson(s, Id, alpha)
    got = api.emfuse_backward(g.to(dev), f, s, Id, *sigmas, alpha)
    x, gd = I0.double().numpy(), g.double().numpy()
    dI0, _, dsig = O.backward_stack(gd, x, *sigmas, alpha)
    lam = np.stack([O.apply_Ainv(gj, alpha) for gj in gd])
    lap = O.laplacian(lam)
    assert np.abs(got["in0"].cpu().numpy() - dI0).max() <= 1e-4 * np.abs(dI0).max()
    assert np.abs(got["o"].cpu().numpy() - lap).max() <= 1e-4 * max(np.abs(lap).max(), 1e-6 * np.abs(lam).max())
    dk = O.dsmooth_dsigma_z(x, *sigmas)
    assert abs(got["sigma_z"] - dsig) <= 1e-4 * np.abs(alpha * lam * dk).sum()


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("cell", [(0, 0, 0), (12, 20, 16), (23, 39, 32), (11, 8, 31)])
def test_values_that_are_not_finite_stay_in_their_support(dev, value, cell):
    """A tap outside the support never meets them: cells beyond it are what they are without."""
    I0 = make_stack(24, 40, 33, seed=2).to(dev)
    sigmas, R = (3.0, 1.0), (3, 9, 9)
    I0[cell] = 0.0
    ref = api.emfuse_smooth_z(I0, *sigmas)
    I0[cell] = value
    out = api.emfuse_smooth_z(I0, *sigmas)
    inside = torch.zeros(out.shape, dtype=torch.bool, device=dev)
    inside[tuple(slice(max(0, c - r), c + r + 1) for c, r in zip(cell, R))] = True
    assert not torch.isfinite(out[inside]).any()
    assert torch.equal(out[~inside], ref[~inside])
