"""A state uploaded from host memory, array by array, against the same state set
from device memory in one launch: the arrays, the wave speed that came with the
load, and the steps from its ghost layers, bit for bit."""
import numpy as np
import pytest

from paper_2508_06273_gb300 import workloads as W
from test_gpu_parity import env, solver, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu
SIDES = {"periodic": (0, 0, 0, 0), "outflow": (1, 1, 1, 1), "walls": (2, 2, 2, 2), "inflow": (3, 1, 2, 3)}


@pytest.mark.parametrize("asynchronous", [False, True])
@pytest.mark.parametrize("sides", SIDES)
@pytest.mark.parametrize("nx,ny", [(2, 2), (31, 33), (70, 29)])
def test_host_upload_equals_device_load(env, nx, ny, sides, asynchronous):  # noqa: F811
    torch = env[0]
    p = W.fourier_smooth(nx, ny, seed=8, lx=0.1 * nx, ly=0.1 * ny, amp=0.05, modes=2)
    p.bc = SIDES[sides]
    if sides == "inflow":
        p.inflow = {0: (1.0, 0.3, -0.2, 1.0), 3: (1.1, 0.2, -0.1, 1.2)}
    first, st = [W.to_f32(W.discretise(p)) for _ in range(2)]
    st = [np.ascontiguousarray(a * np.float32(1.01), dtype=np.float32) for a in st]
    a, b = solver(env, p, state=first), solver(env, p, state=st)
    a.step(0.1 * min(p.dx, p.dy) / a.max_speed())  # leaves low words, status and ghosts to replace
    (a.set_state_host_async if asynchronous else a.set_state)(*st)  # (arrays on the host)
    assert a.max_speed() == b.max_speed()
    dt = 0.2 * min(p.dx, p.dy) / b.max_speed()
    for k in range(3):
        for x, y in zip([*a.get_state(), a.get_avg_lo()], [*b.get_state(), b.get_avg_lo()]):
            assert torch.equal(x, y), k
        assert a.status() == b.status() and a.max_speed() == b.max_speed()
        a.step(dt)
        b.step(dt)
    a.host_sync()
    a.close()
    b.close()
