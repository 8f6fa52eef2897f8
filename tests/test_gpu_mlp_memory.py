"""Training with a batch whose scratch cannot be allocated is refused, and what
the handle held before is given back: the next calls allocate what they need
again instead of using it."""
import numpy as np
import pytest

from test_gpu_mlp import _data, lib, net  # noqa: F401

pytestmark = pytest.mark.gpu
IMPOSSIBLE = 2 ** 31 - 8  # 1696 bytes a row: 3.6 TB


@pytest.mark.parametrize("first", ["forward", "loss_grad", "train"])
def test_calls_after_a_refused_batch(lib, net, first):  # noqa: F811
    torch, _ = lib
    from paper_2508_06273_gb300 import af

    m, p = net
    X, T, Xd, Td = _data(torch, 300, 12)
    want = {"forward": m.forward(Xd), "loss_grad": m.loss_grad(Xd, Td), "train": m.train(Xd, Td, 2, batch=64)}
    m.set_params(p)
    with pytest.raises(af.AFError, match="scratch"):
        m.train(Xd, Td, 1, batch=IMPOSSIBLE)
    m.set_params(p)  # (Adam's step count too)
    for call in [first] + [c for c in want if c != first]:
        if call == "forward":
            assert torch.equal(m.forward(Xd), want[call])
        elif call == "loss_grad":
            loss, grads = m.loss_grad(Xd, Td)
            assert loss == want[call][0] and np.array_equal(grads, want[call][1])
        else:
            assert np.array_equal(m.train(Xd, Td, 2, batch=64), want[call])
            m.set_params(p)
