"""The kernels a level can run by (coarse tail, tiles, wavefronts) against the reference schedule
(one kernel per half-sweep), bit for bit, at the sizes where each can go wrong: the 64-cell edge of
the tail and levels of few cells, tile edges (outputs of 112 / 120 columns and 52 / 56 rows for two
sweeps), partial cells on either axis, and batches on both sides of the line between tiles and
wavefronts (5 M cells in FP32, 2.5 M in FP64), whose strips are of widths that are not multiples of 4."""
import pytest
import torch

from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu

TAIL = [(2, 1, 64), (2, 64, 1), (3, 2, 2), (2, 3, 61), (2, 64, 64), (1, 63, 33)]
TILE = [(1, 65, 66), (2, 52, 112), (1, 53, 113), (2, 56, 120), (1, 57, 121), (1, 105, 225), (2, 67, 3), (1, 1, 241),
        (1, 241, 1), (1, 700, 130)]
WAVE = [(1, 2301, 2211), (5, 1031, 1026), (1, 1100, 5003), (2, 2050, 1605)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch.device("cuda", 0)


def both(dev, shape, nu, precision):
    g = torch.Generator(device=dev).manual_seed(7)
    s = 255.0 * torch.rand(shape, generator=g, device=dev)
    o = 0.9 * s + 20.0 * torch.rand(shape, generator=g, device=dev)
    out = []
    for fused in (1, 0):
        opts = api.default_opts(fused=fused, nu_pre=nu[0], nu_post=nu[1], precision=precision, max_vcycles=3, tol=0.0)
        out.append(api.emfuse_screened_poisson(s, o, 1e-3, opts, allow_noconv=True))
    return out


@pytest.mark.parametrize("shape", TAIL + TILE)
@pytest.mark.parametrize("nu", [(2, 2), (1, 3), (3, 1)])
@pytest.mark.parametrize("precision", [api.PREC_MIXED, api.PREC_FP64])
def test_tail_and_tiles_equal_the_reference_schedule(dev, shape, nu, precision):
    a, b = both(dev, shape, nu, precision)
    assert torch.equal(a, b)


@pytest.mark.parametrize("shape", WAVE)
@pytest.mark.parametrize("nu", [(2, 2), (3, 4)])
@pytest.mark.parametrize("precision", [api.PREC_MIXED, api.PREC_FP64])
def test_wavefronts_equal_the_reference_schedule(dev, shape, nu, precision):
    a, b = both(dev, shape, nu, precision)
    assert torch.equal(a, b)
