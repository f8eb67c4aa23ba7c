"""Single-column stencils on vectors that are 8-byte aligned only: the layouts that read element by element keep
their choice, and only the bulk-copy kernel gives way to the register kernel.  Every layout sums in a fixed order,
so the route shows in the bits."""
import pytest
import torch

from test_gpu_digits import blocks, columns
from test_gpu_mcol import operator
from test_gpu_site8 import fixed, unaligned

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,nv", [((2, 3, 2, 2), 8), ((2, 2, 2, 5), 16), ((4, 2, 2, 2), 24)])
@pytest.mark.parametrize("prec", [1, 2])
def test_choice_is_kept(dims, nv, prec):
    s, f = blocks(dims, nv, 81)
    V, n = s.shape[0], 2 * nv
    x = torch.from_numpy(columns(1, V * n, 82)[0]).cuda().to(torch.complex64)
    x8 = unaligned(x)
    assert x.data_ptr() % 16 == 0 and x8.data_ptr() % 16 == 8
    dev = operator(s, f, dims, nv, 0.02, 1)
    out = {}
    for choice in (1, 2):
        with fixed("apply", n, V, choice):
            out[choice] = dev.apply(x, precision=prec)
            assert torch.equal(dev.apply(x8, precision=prec), out[choice])
        with fixed("apply", n, V, choice):  # the choice first met with an unaligned vector
            assert torch.equal(dev.apply(x8, precision=prec), out[choice])
    with fixed("apply", n, V, 0):
        assert torch.equal(dev.apply(x8, precision=prec), out[1])
    assert not torch.equal(out[1], out[2])
    dev.close()
