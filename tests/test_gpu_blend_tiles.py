"""The blend weights, formed tile by tile (32 x 8 edges with the cells around
them), at sizes around the tiles and with every kind of side: one step with the
blend against the oracle, and a batch's against the single grid's bit for bit."""
import pytest

from helpers import make_oracle
from paper_2508_06273_gb300 import workloads as W
from test_gpu_parity import STEP_TOL, assert_parity, env, host, solver, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu
SIDES = {"periodic": (0, 0, 0, 0), "outflow": (1, 1, 1, 1), "walls": (2, 2, 2, 2), "mixed": (1, 2, 0, 0)}


@pytest.mark.parametrize("sides", SIDES)
@pytest.mark.parametrize("nx,ny", [(3, 2), (30, 6), (31, 8), (33, 7), (62, 17)])
def test_blend_at_tile_edges(env, nx, ny, sides):  # noqa: F811
    torch, af, oracle = env
    p = W.fourier_smooth(nx, ny, seed=8, lx=0.1 * nx, ly=0.1 * ny, amp=0.2, modes=2)
    p.bc = SIDES[sides]
    p.options = {"shock_blend": 1}
    st = W.to_f32(W.discretise(p))
    o, s = make_oracle(oracle, p, state=st), solver(env, p, state=st)
    b = af.Batch([(nx, ny)], [(p.dx, p.dy)], bcs=[p.bc])
    b.set_option("shock_blend", 1, 0)
    b.set_state(0, *to_dev(torch, st))
    b.set_end(float("inf"), 0.2)
    hist = torch.zeros((1, 1), dtype=torch.float64, device="cuda")
    b.run(1, hist)
    dt = float(hist[0, 0])
    o.step(dt)
    s.step(dt)
    assert_parity(host(s.get_state()), o.get_state(), STEP_TOL, what=f"{nx}x{ny} {sides}")
    assert all(torch.equal(x, y) for x, y in zip(b.get_state(0), s.get_state()))
    b.close()
