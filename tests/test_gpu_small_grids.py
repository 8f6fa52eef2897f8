"""Small grids, whose steps take the split point-value tiles and the flux
kernel that fills the ghost entries itself: sizes at the edges of the tiles and
of the ghost layers, every kind of side, against the oracle; and the pieces that
carry state from one step to the next (ghosts, counters, wave speed) against a
handle that starts anew from each step's state."""
import numpy as np
import pytest

from helpers import make_oracle
from paper_2508_06273_gb300 import workloads as W
from test_gpu_parity import assert_parity, env, host, solver, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu
SIDES = {"periodic": (0, 0, 0, 0), "outflow": (1, 1, 1, 1), "walls": (2, 2, 2, 2), "mixed": (1, 2, 0, 0),
         "inflow": (3, 1, 2, 3)}


def _problem(nx, ny, sides):
    p = W.fourier_smooth(nx, ny, seed=8, lx=0.1 * nx, ly=0.1 * ny, amp=0.05, modes=2)
    p.bc = SIDES[sides]
    if sides == "inflow":
        p.inflow = {0: (1.0, 0.3, -0.2, 1.0), 3: (1.1, 0.2, -0.1, 1.2)}
    return p


@pytest.mark.parametrize("sides", SIDES)
@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 2), (2, 9), (31, 4), (32, 8), (33, 5), (65, 17)])
def test_steps_match_the_oracle(env, nx, ny, sides):  # noqa: F811
    torch, af, oracle = env
    p = _problem(nx, ny, sides)
    st = W.to_f32(W.discretise(p))
    o, s = make_oracle(oracle, p, state=st), solver(env, p, state=st)
    dt = 0.2 * min(p.dx, p.dy) / o.max_speed()
    for _ in range(3):
        o.step(dt)
        s.step(dt)
        assert s.max_speed() == pytest.approx(o.max_speed(), rel=1e-5)
    assert_parity(host(s.get_state()), o.get_state(), 3e-5, what=f"{nx}x{ny} {sides}")


@pytest.mark.parametrize("sides", SIDES)
def test_a_step_carries_what_a_new_handle_computes(env, sides):  # noqa: F811
    torch, af, _ = env
    p = _problem(45, 21, sides)
    p.options = {"tsw": 1, "flux_limiter": 1, "shock_blend": 1, "node_bounds": 1, "ubar": 1}
    s = solver(env, p)
    dt = 0.2 * min(p.dx, p.dy) / s.max_speed()
    for k in range(4):
        fresh = solver(env, p, state=None)
        fresh.set_state(*s.get_state())
        fresh.set_avg_lo(s.get_avg_lo())
        s.step(dt)
        fresh.step(dt)
        for a, b in zip(s.get_state(), fresh.get_state()):
            assert torch.equal(a, b), k
        assert s.counters() == fresh.counters() and s.max_speed() == fresh.max_speed(), k


def test_run_from_either_buffer_equals_steps(env):  # noqa: F811
    torch, af, _ = env
    p = _problem(40, 13, "mixed")
    a, b = solver(env, p), solver(env, p)
    dt = 0.2 * min(p.dx, p.dy) / a.max_speed()
    for n in (4, 5, 6, 7):  # odd counts change the buffer the next run starts from
        a.run(n, dt)
        for _ in range(n):
            b.step(dt)
        for x, y in zip(a.get_state(), b.get_state()):
            assert torch.equal(x, y), n
        assert a.max_speed() == b.max_speed() and a.counters() == b.counters()
