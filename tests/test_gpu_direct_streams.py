"""The direct solvers on streams other than the default one: the first call of a size, which forms
the plan's tables, gives what later calls on other streams give."""
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


def on(stream, fn):
    with torch.cuda.stream(stream):
        return fn()


# slices of a few cells under tables of up to 4 MB (the z matrix), and long rows
@pytest.mark.parametrize("shape", [(1009, 5, 7), (300, 3, 2), (2, 3, 40009), (5, 255, 129)])
@pytest.mark.parametrize("precision", [api.PREC_FP32, api.PREC_FP64])
def test_first_call_of_a_size(dev, shape, precision):
    I0 = torch.from_numpy(np.random.default_rng(21).uniform(0, 255, size=shape).astype(np.float32)).to(dev)
    o = (0.9 * I0 + 10).contiguous()
    torch.cuda.synchronize()
    side = [torch.cuda.Stream(), torch.cuda.Stream()]
    for call in (lambda: api.emfuse_screened_poisson_dct(I0, o, 0.01, precision),
                 lambda: api.emfuse_smooth_gradient_domain(I0, 0.05, precision)):
        api.lib().emfuse_release_cache()
        first = on(side[0], call)
        again = on(side[1], call)
        torch.cuda.synchronize()
        assert torch.equal(first, again)
        assert torch.equal(first, call())
