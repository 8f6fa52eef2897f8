"""Sums over batches of several tiles a CTA, on inputs whose exact sums a short
chain of FP32 additions would lose: all weights zero, so that the output is zero
and the squared errors are powers of two."""
import numpy as np
import pytest

from test_gpu_mlp import lib  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture
def zero_net(lib):  # noqa: F811
    from paper_2508_06273_gb300 import af

    m = af.Mlp(seed=1)
    p = np.zeros_like(m.get_params())
    p[43408:] = 1.0  # input and output scales
    m.set_params(p)
    yield lib[0], m, p
    m.close()


def test_loss_of_many_tiles_is_summed_in_64_bits(zero_net):
    torch, m, _ = zero_net
    half = 128 * torch.cuda.get_device_properties(0).multi_processor_count
    T = torch.ones((2 * half, 8), device="cuda")
    T[:half] = 2.0 ** 13  # every CTA's first tile: its 32-row sums, 2^34, have an FP32 step of 2^11
    X = torch.zeros((2 * half, 64), device="cuda")
    loss, _ = m.loss_grad(X, T)
    # the squares and 32-row sums are exact; a handful of roundings in 64 bits remain
    assert loss == pytest.approx((2.0 ** 26 + 1) / 2, rel=1e-12)
