"""The correction passes of large mixed-precision batches form A d from FP64 values split into two
floats (batches of 16 M cells and more) instead of in FP64: both against the 64-bit solution, and
against each other through the batch size, which selects the form.  A solve of the same slice
inside a batch below and above the line differs only by the rounding of A d, at most an ulp of it
per pass (2^-24 |A d|, alpha |d| and smaller), which A^-1 can amplify by 1 / alpha at most: 2^-23 of
the largest |d|, with the rounding of the FP32 output on top."""
import numpy as np
import pytest
import torch

from oracle import emfuse_oracle as O
from paper_1506_02079_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch.device("cuda", 0)


# one slice of each shape, repeated until the batch has 16 M cells: tiles of 64 x 32 with remainders,
# a narrow slice, a multiple of the tile (no interior tile touches its last row or column)
@pytest.mark.parametrize("shape", [(1021, 1027), (4100, 33), (1024, 2048), (31, 5003)])
@pytest.mark.parametrize("alpha", [1e-3, 0.1])
def test_split_form_matches_fp64_form(dev, shape, alpha):
    ny, nx = shape
    rng = np.random.default_rng(4)
    yy, xx = np.mgrid[0:ny, 0:nx]
    s = (128 + 60 * np.sin(yy / 37.0) * np.cos(xx / 53.0) + rng.uniform(-20, 20, size=shape)).astype(np.float32)
    o = np.clip(0.9 * s + 15 * np.cos(xx / 91.0), 0, 255).astype(np.float32)
    n = -(-16_000_000 // (ny * nx))
    opts = api.default_opts(tol=2e-7)
    st, ot = torch.from_numpy(s).to(dev), torch.from_numpy(o).to(dev)
    one, s1 = api.emfuse_screened_poisson(st[None].contiguous(), ot[None].contiguous(), alpha, opts, return_stats=True)
    many, sn = api.emfuse_screened_poisson(st.expand(n, ny, nx).contiguous(), ot.expand(n, ny, nx).contiguous(), alpha,
                                           opts, return_stats=True)
    assert all(a["converged"] and a["vcycles"] == s1[0]["vcycles"] for a in sn)
    assert torch.equal(many[0], many[-1])
    passes = s1[0]["vcycles"]
    ref = O.solve_dct(s.astype(np.float64), o.astype(np.float64), alpha)
    dmax = float(np.abs(ref - o).max())
    bar = passes * 2.0 ** -23 * dmax + 2.0 ** -16  # an ulp of the output below 256
    assert float((many[0] - one[0]).abs().max()) <= bar
    e1 = float(np.linalg.norm(one[0].cpu().double().numpy() - ref))
    en = float(np.linalg.norm(many[0].cpu().double().numpy() - ref))
    assert en <= 1.001 * e1
