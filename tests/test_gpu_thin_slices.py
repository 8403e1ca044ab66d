"""Levels of few cells whose tiles would be nearly empty (slices of a few rows or columns, many slices
just above the coarse tail's size) run by wavefronts: bit for bit the reference schedule, on sizes
on either side of the line (twice 5 M cells in tiles of 128 x 64, FP64 twice 2.5 M in 128 x 32)."""
import pytest
import torch

from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 136000), (1, 1, 137000), (1, 3, 150001), (2, 70, 60000), (1, 70001, 1), (1, 62000, 5),
                                   (620, 65, 66), (600, 65, 66), (1, 33, 140003)])
@pytest.mark.parametrize("precision", [api.PREC_MIXED, api.PREC_FP64])
def test_equal_to_the_reference_schedule(shape, precision):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    dev = torch.device("cuda", 0)
    g = torch.Generator(device=dev).manual_seed(7)
    s = torch.rand(shape, generator=g, device=dev) * 255
    o = 0.9 * s + 25 * torch.rand(shape, generator=g, device=dev)
    kw = {"precision": precision, "max_vcycles": 3}
    f, st = api.emfuse_screened_poisson(s, o, 0.01, api.default_opts(**kw), return_stats=True, allow_noconv=True)
    r, sr = api.emfuse_screened_poisson(s, o, 0.01, api.default_opts(fused=0, **kw), return_stats=True, allow_noconv=True)
    assert torch.equal(f, r)
    assert [a["rel_residual"] for a in st] == pytest.approx([a["rel_residual"] for a in sr], rel=1e-6)
