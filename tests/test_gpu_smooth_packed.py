"""Smoothing of stacks whose rows TMA cannot read (a byte pitch or base address that is no multiple
of 16) through packed slabs: bit-identical to the plain-load kernel, which emfuse_smooth_z_noalloc
runs, at tile edges (64 columns, 16 rows), for both tap counts along z, for z ranges, pitches and
unaligned bases, with NaN and infinities in the stack, and for stacks packed in several slabs of rows."""
import ctypes

import pytest
import torch

from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch.device("cuda", 0)


def stack(dev, shape, dtype, seed=3):
    g = torch.Generator(device=dev).manual_seed(seed)
    return torch.randint(0, 256, shape, generator=g, device=dev).to(dtype)


def plain(x, sxy, sz, z0=0, z1=None):
    z1 = x.shape[0] if z1 is None else z1
    out = torch.empty((z1 - z0,) + tuple(x.shape[1:]), device=x.device, dtype=torch.float32)
    return api.emfuse_smooth_z_noalloc(x, sxy, sz, out, z0, z1)


@pytest.mark.parametrize("shape", [(5, 17, 33), (1, 1, 1), (23, 70, 9), (12, 16, 65), (21, 33, 127), (3, 15, 63), (4, 100, 203)])
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
@pytest.mark.parametrize("sig", [(1.0, 3.0), (0.5, 1.0), (1.4, 2.5), (0.8, 0.5)])
def test_equals_the_plain_load_kernel(dev, shape, dtype, sig):
    x = stack(dev, shape, dtype)
    assert torch.equal(api.emfuse_smooth_z(x, *sig), plain(x, *sig))
    if shape[0] > 4:
        assert torch.equal(api.emfuse_smooth_z(x, *sig, z0=2, z1=shape[0] - 1), plain(x, *sig, 2, shape[0] - 1))


@pytest.mark.parametrize("sz", [1.0, 3.0])
def test_non_finite_values_spread_as_far(dev, sz):
    x = stack(dev, (30, 40, 51), torch.float32)
    x[11, 20, 25] = float("nan")
    x[22, 3, 50] = float("inf")
    a, b = api.emfuse_smooth_z(x, 1.0, sz), plain(x, 1.0, sz)
    assert torch.equal(torch.nan_to_num(a, nan=-1.0, posinf=-2.0), torch.nan_to_num(b, nan=-1.0, posinf=-2.0))


@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
def test_unaligned_base_with_an_aligned_pitch(dev, dtype):
    nz, ny, nx = 9, 40, 64
    flat = stack(dev, (nz * ny * nx + 1,), dtype)
    x = flat[1:].view(nz, ny, nx)  # rows of 64 elements that start one element past a 16-byte boundary
    assert torch.equal(api.emfuse_smooth_z(x, 1.0, 3.0), plain(x, 1.0, 3.0))


def test_pitch_beyond_the_row(dev):
    nz, ny, nx, pitch = 6, 30, 61, 67
    wide = stack(dev, (nz, ny, pitch), torch.float32)
    out = torch.full((nz, ny, pitch), -7.0, device=dev)
    code = api.lib().emfuse_smooth_z(wide.data_ptr(), api.EMFUSE_F32, out.data_ptr(), nx, ny, nz, pitch, 0, nz,
                                     ctypes.c_float(1.0), ctypes.c_float(3.0),
                                     torch.cuda.current_stream(dev).cuda_stream)
    assert code == 0
    assert torch.equal(out[:, :, :nx], plain(wide[:, :, :nx].contiguous(), 1.0, 3.0))
    assert bool((out[:, :, nx:] == -7.0).all())


def test_several_slabs(dev):
    x = stack(dev, (600, 1100, 1021), torch.uint8)  # 614 KB per row of all planes: slabs of 864 rows
    assert torch.equal(api.emfuse_smooth_z(x, 1.0, 3.0), plain(x, 1.0, 3.0))
