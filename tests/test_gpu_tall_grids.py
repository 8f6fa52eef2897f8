"""Grids of more rows than 65535 blocks of the plain kernels' 4-row tiles cover:
the library picks a taller tile, with the results of 8-row tiles set by hand, bit
for bit, in single steps and captured runs."""
import numpy as np
import pytest

from paper_2508_06273_gb300 import workloads as W
from test_gpu_parity import env, solver  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("options", [{}, {"lin_mode": 2}], ids=["plain", "two_stage"])
@pytest.mark.parametrize("ny", [262139, 262140])  # node rows 262140 = 4 x 65535, and one more
def test_tall_grids_step(env, ny, options):  # noqa: F811
    torch = env[0]
    p = W.fourier_smooth(2, 64, seed=8, lx=0.2, ly=6.4, amp=0.05, modes=2)
    short = W.to_f32(W.discretise(p))
    p.ny, p.bc, p.options = ny, (1, 1, 1, 1), options
    # the 64-row data repeated along y (its first and last node lines agree)
    st = [np.ascontiguousarray(a[:, np.arange(n) % 64]) for a, n in zip(short, (ny, ny + 1, ny, ny + 1))]
    a, b = solver(env, p, state=st), solver(env, p, state=st)
    b.set_option("tile_h", 8)
    dt = 0.2 * min(p.dx, p.dy) / a.max_speed()
    for s in (a, b):
        s.step(dt)
        s.run(4, dt)
    assert a.status() == b.status() == 0 and a.max_speed() == b.max_speed()
    for x, y in zip([*a.get_state(), a.get_avg_lo()], [*b.get_state(), b.get_avg_lo()]):
        assert torch.equal(x, y)
    a.close()
    b.close()
