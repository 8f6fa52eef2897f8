"""The reductions that leave their result in host memory in one launch (totals,
minima, wave speed) and the small results a step hands over (status, counters),
at sizes around the tiles that a block reduces, against NumPy in double precision."""
import numpy as np
import pytest

from paper_2508_06273_gb300 import workloads as W
from test_gpu_parity import env, host, solver, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


def _values(state, gamma=1.4):
    """Primitive states of the averages and of the owned point values."""
    q = state[0].astype(np.float64)
    rho, u, v = q[0], q[1] / q[0], q[2] / q[0]
    avg = np.stack([rho, u, v, (gamma - 1) * (q[3] - 0.5 * rho * (u * u + v * v))])
    return [avg] + [a.astype(np.float64) for a in state[1:]]


@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 1, 2, 2)])
@pytest.mark.parametrize("nx,ny", [(2, 2), (31, 7), (32, 8), (33, 9), (65, 300), (700, 611)])
def test_reductions_match_numpy(env, nx, ny, bc):  # noqa: F811
    p = W.fourier_smooth(nx, ny, seed=4, lx=0.1 * nx, ly=0.1 * ny, amp=0.05, modes=2)
    p.bc = bc
    s = solver(env, p)
    dt = 0.2 * min(p.dx, p.dy) / s.max_speed()
    for k in range(3):
        arrays = host(s.get_state())
        U = _values(arrays)
        # the FP32 conversion of an average: a few roundings of 6e-8
        assert s.state_min() == pytest.approx((min(a[0].min() for a in U), min(a[3].min() for a in U)), rel=1e-6)
        speed = max((np.maximum(abs(a[1]), abs(a[2])) + np.sqrt(1.4 * a[3] / a[0])).max() for a in U)
        assert s.max_speed() == pytest.approx(speed, rel=2e-6)
        lo = host([s.get_avg_lo()])[0].astype(np.float64)
        q = arrays[0].astype(np.float64) + lo
        want = q.sum(axis=(1, 2)) * p.dx * p.dy
        # the same doubles summed in another order
        np.testing.assert_allclose(s.totals(), want, rtol=0, atol=1e-12 * abs(q).sum() * p.dx * p.dy)
        assert s.totals().tobytes() == s.totals().tobytes()
        s.step(dt) if k else s.run(6, dt)
        assert s.status() == 0


@pytest.mark.parametrize("n", [24, 1700])
def test_status_and_counters_by_either_way(env, n):  # noqa: F811
    """A small grid's step hands them over; after the state is set anew, and on a
    large grid, they are fetched."""
    af = env[1]
    p = W.four_quadrant(n, seed=5)
    s = solver(env, p)
    assert s.counters() == [0, 0, 0, 0]
    dt = 0.2 * min(p.dx, p.dy) / s.max_speed()
    s.step(dt)
    c, state = s.counters(), s.get_state()
    assert sum(c) > 0 and not s.status() & af.ST_CFL
    s.set_state(*state)
    assert s.counters() == c and s.status() == 0
    s.step(15 * dt)  # CFL 3: the cone base leaves the stencil
    assert s.status() & af.ST_CFL and s.status() == 0
    s.step(15 * dt)
    s.set_state(*state)
    assert s.status() == 0
    s.run(6, dt)
    assert not s.status() & af.ST_CFL
