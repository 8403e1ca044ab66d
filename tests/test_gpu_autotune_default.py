"""The autotuner times the default schedule (heights chosen by the library, nu = (2, 2)) among its
candidates, so the schedule it takes is never slower by its own clock."""
import pytest
import torch

from paper_1506_02079_gb300 import api
from paper_1506_02079_gb300.synthetic import make_ragged_batch

pytestmark = pytest.mark.gpu


def test_default_is_a_candidate():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    dev = torch.device("cuda", 0)
    s, o, ny, nx, offs = make_ragged_batch(6, seed=3, side_lo=900, side_hi=1900)
    s, o = s.to(dev), o.to(dev)
    f = api.emfuse_screened_poisson(s, o, 1e-3, api.default_opts(autotune=1), nx=nx, ny=ny, offsets=offs)
    table = api.emfuse_autotune_result()
    default = [e for e in table if (e["nu_pre"], e["nu_post"], e["tile_rows"]) == (2, 2, 0)]
    assert len(default) == 1 and table[0]["ms"] <= default[0]["ms"]
    best = api.default_opts(nu_pre=table[0]["nu_pre"], nu_post=table[0]["nu_post"], tile_rows=table[0]["tile_rows"])
    assert torch.equal(f, api.emfuse_screened_poisson(s, o, 1e-3, best, nx=nx, ny=ny, offsets=offs))
