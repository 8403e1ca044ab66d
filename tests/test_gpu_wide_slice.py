"""A slice so wide that 32 rows of it span more than 2^31 cells: the residual passes reach up to 32 rows
beyond a tile's corner, so their offsets need 64 bits there.  s - o is one cosine mode along y
(the same in every column), whose solution is known in closed form at every cell:
f = o + alpha / (alpha + lambda) (s - o), lambda = 4 sin^2(pi / 2 ny)."""
import math

import pytest
import torch

from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu

NX, NY = 1 << 26, 33  # row 32 of the first tile starts 2^31 cells from its corner
NEEDED = 125e9        # s, o, f, the pyramid and two FP64 iterates: 50 B per cell, with some room


def test_offsets_beyond_31_bits():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda", 0)
    torch.cuda.empty_cache()
    api.lib().emfuse_release_cache()
    if torch.cuda.mem_get_info(dev)[0] < NEEDED:
        pytest.skip("needs 125 GB of free device memory")
    alpha = 0.1
    mode = 60.0 * torch.cos(math.pi * (torch.arange(NY, dtype=torch.float64) + 0.5) / NY)
    gain = alpha / (alpha + 4.0 * math.sin(math.pi / (2 * NY)) ** 2)
    level = torch.linspace(100.0, 140.0, NY, dtype=torch.float64)
    o = level.float().to(dev)[:, None].expand(NY, NX).contiguous()
    s = (level + mode).float().to(dev)[:, None].expand(NY, NX).contiguous()
    try:
        f, st = api.emfuse_screened_poisson(s[None], o[None], alpha, return_stats=True)
        assert st[0]["converged"]
        exact = (level + gain * mode).float().to(dev)
        # ||f - f*|| <= ||r|| / alpha bounds the sum over all cells only; the error follows the mode, so a
        # cell's share is the mean, taken ten times, with an ulp of the output
        bar = 10.0 * st[0]["rel_residual"] * st[0]["b_norm"] / alpha / math.sqrt(NX * NY) + 2.0 ** -16
        for y in range(NY):
            assert float((f[0, y] - exact[y]).abs().max()) <= bar, y
    finally:
        del s, o
        f = None
        torch.cuda.empty_cache()
        api.lib().emfuse_release_cache()
