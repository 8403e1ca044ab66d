"""A slice's result does not depend on what it is solved with: whole stacks on the device, both host
pipelines, a shard and single slices give the same bits.  Totals of 20 M cells in chunks of a few
million, with slices on either side of the size from which A d is formed in split form (a million
cells), and a ragged batch with both kinds."""
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


def stack(dev, shape, seed):
    nz, ny, nx = shape
    g = torch.Generator(device=dev).manual_seed(seed)
    y = torch.arange(ny, device=dev)[None, :, None] / 37.0
    x = torch.arange(nx, device=dev)[None, None, :] / 53.0
    z = torch.arange(nz, device=dev)[:, None, None] * 2.1
    return 128 + 60 * torch.sin(y) * torch.cos(x + 0.3 * z) + 15 * torch.sin(z) + 20 * torch.rand(shape, generator=g, device=dev)


@pytest.mark.parametrize("shape", [(20, 1024, 1024), (80, 512, 511), (9, 1187, 2001)])
def test_host_pipelines_equal_the_device(dev, shape):
    I0 = stack(dev, shape, 3).clamp(0, 255)
    f, st = api.emfuse_correct_stack(I0, return_stats=True)
    host = I0.cpu().pin_memory()
    for kw in ({"host_pipeline": 2}, {"host_pipeline": 1, "host_chunk": 3}):
        h, sh = api.emfuse_correct_stack(host, opts=api.default_opts(**kw), return_stats=True)
        assert torch.equal(h, f.cpu()), kw
        assert [a["vcycles"] for a in sh] == [a["vcycles"] for a in st]


def test_groups_equal_single_slices(dev):
    sides = [(300, 401), (999, 1001), (1000, 1000), (1001, 999), (64, 64), (4000, 4001), (33, 40000), (2000, 3)]
    s, o = [], []
    for j, (ny, nx) in enumerate(sides):
        a = stack(dev, (2, ny, nx), j)
        s.append(a[0].contiguous())
        o.append(a[1].contiguous())
    many, st = api.emfuse_screened_poisson(s, o, 1e-3, return_stats=True)
    for j in range(len(sides)):
        one, s1 = api.emfuse_screened_poisson(s[j], o[j], 1e-3, return_stats=True)
        assert torch.equal(one, many[j]), sides[j]
        assert s1[0]["vcycles"] == st[j]["vcycles"]
