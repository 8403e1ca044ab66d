"""Smoothing of unaligned rows over one to three planes, by plain loads or packed on either side of the
line (400,000 cells of input): the plain-load kernel's bits (emfuse_smooth_z_noalloc), and for robust
averaging those of the same planes with their rows several times over, which is packed."""
import pytest
import torch

from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu

SHAPES = [(1, 33, 35), (1, 631, 633), (1, 633, 633), (2, 447, 447), (2, 449, 447), (3, 365, 365), (3, 367, 365), (4, 35, 33)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch.device("cuda", 0)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
@pytest.mark.parametrize("sig", [(1.0, 3.0), (0.5, 0.5)])
def test_same_bits_on_either_side(dev, shape, dtype, sig):
    g = torch.Generator(device=dev).manual_seed(13)
    x = torch.randint(0, 256, shape, generator=g, device=dev).to(dtype)
    out = torch.empty(shape, device=dev, dtype=torch.float32)
    assert torch.equal(api.emfuse_smooth_z(x, *sig), api.emfuse_smooth_z_noalloc(x, *sig, out))


@pytest.mark.parametrize("shape", [(1, 40, 35), (2, 447, 447), (3, 40, 35)])
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
def test_robust(dev, shape, dtype):
    nz, ny, nx = shape
    g = torch.Generator(device=dev).manual_seed(14)
    x = torch.randint(0, 256, shape, generator=g, device=dev).to(dtype)
    f = api.emfuse_smooth_z_robust(x, 1.0, 3.0, 2.0)
    # rows away from the seams have the same neighbours
    h = api.emfuse_smooth_z_robust(x.repeat(1, 300000 // (ny * nx) + 2, 1).contiguous(), 1.0, 3.0, 2.0)
    assert torch.equal(f[:, :ny - 3], h[:, :ny - 3])
    assert torch.equal(f[:, 3:], h[:, -ny + 3:])
