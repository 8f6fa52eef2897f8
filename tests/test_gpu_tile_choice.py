"""The tile that the library picks while none is chosen (split, 4 or 8 rows, by
size and options) gives bit for bit the results of every height that can be set,
on both sides of the rule's lines, for single grids and for batches."""
import pytest

from paper_2508_06273_gb300 import workloads as W
from test_gpu_parity import env, solver, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu
RIEMANN = {"tsw": 1, "flux_limiter": 1, "shock_blend": 1, "node_bounds": 1, "ubar": 1}
OPTIONS = {"plain": {}, "two_stage": {"lin_mode": 2}, "node_flux": {"node_flux": 1}, "riemann": RIEMANN}


@pytest.mark.parametrize("options", OPTIONS)
@pytest.mark.parametrize("nx,ny", [(5, 3), (128, 152), (128, 156), (129, 121), (130, 300)])
def test_choice_equals_every_height(env, nx, ny, options):  # noqa: F811
    torch = env[0]
    p = W.fourier_smooth(nx, ny, seed=8, lx=0.1 * nx, ly=0.1 * ny, amp=0.05, modes=2)
    p.options = OPTIONS[options]
    state, dt = W.to_f32(W.discretise(p)), None
    want = None
    for tile in (None, 4, 8, 16):
        s = solver(env, p, state=state)
        if tile:
            s.set_option("tile_h", tile)
        dt = dt or 0.2 * min(p.dx, p.dy) / s.max_speed()
        s.run(5, dt)
        got = s.get_state()
        want = want or got
        assert all(torch.equal(a, b) for a, b in zip(got, want)), tile
        s.set_option("lin_mode", 2 if options == "plain" else 0)  # the tile follows the options
        s.step(dt)
        s.close()


def test_batch_choice_equals_every_height(env):  # noqa: F811
    torch, af, _ = env
    sizes = [(40, 33), (65, 20), (31, 64)]
    problems = [W.fourier_smooth(nx, ny, seed=k, lx=0.1 * nx, ly=0.1 * ny, amp=0.05, modes=2)
                for k, (nx, ny) in enumerate(sizes)]
    want = None
    for tile in (None, 4, 8, 16):
        b = af.Batch(sizes, [(p.dx, p.dy) for p in problems], bcs=[p.bc for p in problems])
        b.set_option("lin_mode", 2, 1)
        for key, v in RIEMANN.items():
            b.set_option(key, v, 2)
        if tile:
            b.set_tile(tile)
        for k, p in enumerate(problems):
            b.set_state(k, *to_dev(torch, W.to_f32(W.discretise(p))))
        b.set_end(float("inf"), 0.2)
        b.run(4)
        got = [b.get_state(k) for k in range(3)]
        want = want or got
        for k in range(3):
            assert all(torch.equal(x, y) for x, y in zip(got[k], want[k])), (tile, k)
        b.close()
