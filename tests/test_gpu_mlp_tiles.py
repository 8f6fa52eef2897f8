"""The fused training kernels at the edges of their tiles: batches below,
at and beyond one 128-row tile, ones that give a CTA several tiles and a
split several 256-row steps, and inputs whose rows are not 16-byte aligned.

Tolerance: the reference rounds to BF16 where the GPU does, so a product's two
stored factors are each off by at most one BF16 step (2^-8) where FP32 and FP64
round apart: 2^0.5 x 2^-8 = 5.5e-3 in norm."""
import numpy as np
import pytest

from oracle import surrogate as S
from test_gpu_mlp import LAYERS, _bf16, _data, _unpack, lib, net  # noqa: F401

pytestmark = pytest.mark.gpu
TOL = 2 ** 0.5 * 2 ** -8


def _check(gg, go):
    for name, off, shape in LAYERS:
        a, b = gg[off:off + int(np.prod(shape))].reshape(shape).astype(np.float64), go[name]
        rel = np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30)
        assert rel < TOL, (name, rel)


@pytest.mark.parametrize("n", [1, 7, 128, 129, 8200, 20000])
def test_gradient_at_the_edges_of_the_tiles(lib, net, n):  # noqa: F811
    torch, _ = lib
    m, p = net
    X, T, Xd, Td = _data(torch, n, 30 + n)
    P, ins, outs = _unpack(p, True)
    lo, go = S.loss_and_grads(P, _bf16(X * ins), T / outs, rnd=S.bf16_round)
    lg, gg = m.loss_grad(Xd, Td)
    assert lg == pytest.approx(lo, rel=TOL)
    _check(gg, go)
    again = m.loss_grad(Xd, Td)  # sums in a fixed order
    assert again[0] == lg and np.array_equal(again[1], gg)


def test_rows_off_the_16_byte_boundary(lib, net):  # noqa: F811
    torch, _ = lib
    m, p = net
    X, T, Xd, Td = _data(torch, 200, 77)
    buf = torch.empty(200 * 64 + 1, device="cuda")
    buf[1:] = Xd.reshape(-1)
    off = buf[1:].view(200, 64)
    assert off.data_ptr() % 16 == 4
    assert torch.equal(m.forward(off), m.forward(Xd))
    a, b = m.loss_grad(off, Td), m.loss_grad(Xd, Td)
    assert a[0] == b[0] and np.array_equal(a[1], b[1])
