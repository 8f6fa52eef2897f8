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


def test_weight_gradient_of_many_rows_is_summed_in_short_chains(zero_net):
    torch, m, p = zero_net
    p[41216:41344] = 64.0  # b3: gelu(64) = 64 in every hidden unit of the last layer
    m.set_params(p)
    n = 65536  # 32 splits of 2048 rows: in each, one term of 2^8 and 2047 of 2^-22 (2^-7 of its FP32 step)
    t = torch.full((n,), 2.0 ** -10, device="cuda", dtype=torch.float64)
    t[::2048] = 2.0 ** 20
    want = -float((2 * t / (8 * n)).sum()) * 64
    _, g = m.loss_grad(torch.zeros((n, 64), device="cuda"), t.float()[:, None].expand(n, 8).contiguous())
    got = g[41344:41344 + 8 * 128].astype(np.float64)
    # of a split the terms of the large one's own chain of 512 rows may be lost, 511 of
    # them by 2^-30 each; every other addition rounds by at most 2^-24
    assert np.abs(got / want - 1).max() < 512 * 2.0 ** -30 + 2 * 2.0 ** -24
