"""The direct solvers on streams other than the default one: the first call of a size, which forms
the plan's tables, gives what later calls on other streams give, and calls of one size that run at
the same time on several streams (one plan, one handle) give what they give one after another."""
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


# sides with large prime factors, whose transforms need a work area, and a GEMM with few columns
@pytest.mark.parametrize("shape", [(6, 509, 521), (40, 127, 131), (3, 1, 100003), (900, 5, 7)])
@pytest.mark.parametrize("precision", [api.PREC_FP32, api.PREC_FP64])
def test_same_size_on_several_streams_at_once(dev, shape, precision):
    rng = np.random.default_rng(22)
    side = [torch.cuda.Stream() for _ in range(4)]
    s = [torch.from_numpy(rng.uniform(0, 255, size=shape).astype(np.float32)).to(dev) for _ in side]
    o = [(0.9 * a + 10).contiguous() for a in s]
    serial = [api.emfuse_screened_poisson_dct(s[q], o[q], 0.01, precision) for q in range(len(side))]
    serial3 = [api.emfuse_smooth_gradient_domain(s[q], 0.05, precision) for q in range(len(side))]
    torch.cuda.synchronize()
    got = [on(side[q % 4], lambda: api.emfuse_screened_poisson_dct(s[q % 4], o[q % 4], 0.01, precision)) for q in range(24)]
    got3 = [on(side[q % 4], lambda: api.emfuse_smooth_gradient_domain(s[q % 4], 0.05, precision)) for q in range(24)]
    torch.cuda.synchronize()
    for q in range(24):
        assert torch.equal(got[q], serial[q % 4])
        assert torch.equal(got3[q], serial3[q % 4])
