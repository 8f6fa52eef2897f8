"""Launches that begin while the one before them still writes, over chains of
steps: whole runs against the same steps with the device idle between them, bit
for bit (every sum has a fixed order).  Training at one tile, at several tiles
and at several tiles a CTA; steps on either side of the size up to which the flux
kernel fills the ghosts and hands over the small results (2432 tiles of 32 x 8)."""
import numpy as np
import pytest

from paper_2508_06273_gb300 import workloads as W
from test_gpu_mlp import _data, lib  # noqa: F401
from test_gpu_parity import env, solver, to_dev  # noqa: F401
from test_gpu_small_grids import SIDES, _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [128, 4096, 40000])
def test_training_steps_follow_one_another(lib, batch):  # noqa: F811
    torch, _ = lib
    from paper_2508_06273_gb300 import af

    X, T, Xd, Td = _data(torch, 6000, 5)
    m = af.Mlp(seed=9)
    m.fit_scales(Xd, Td)
    p0 = m.get_params()
    runs = []
    for calls in ([24], [24], [1] * 24):
        m.set_params(p0)
        hist = np.concatenate([m.train(Xd, Td, k, batch=batch, lr=1e-3, seed=3) for k in calls])
        runs.append((hist, m.get_params()))
    assert np.isfinite(runs[0][0]).all() and not np.array_equal(runs[0][1], p0)
    for hist, p in runs[1:]:
        assert np.array_equal(hist, runs[0][0]) and np.array_equal(p, runs[0][1])
    m.close()


@pytest.mark.parametrize("sides", SIDES)
@pytest.mark.parametrize("nx,ny", [(1024, 608), (1025, 609)])
def test_steps_follow_one_another(env, nx, ny, sides):  # noqa: F811
    torch = env[0]
    p = _problem(nx, ny, sides)
    p.options = {"flux_limiter": 1}
    st = W.to_f32(W.discretise(p))
    a, b = solver(env, p, state=st), solver(env, p, state=st)
    dt = 0.2 * min(p.dx, p.dy) / a.max_speed()
    for n in (1, 4, 5):
        a.run(n, dt)
        for _ in range(n):
            fresh = solver(env, p, state=[x.cpu().numpy() for x in b.get_state()])
            fresh.set_avg_lo(b.get_avg_lo())
            b.step(dt)
            torch.cuda.synchronize()
            fresh.step(dt)
            for x, y in zip(b.get_state(), fresh.get_state()):
                assert torch.equal(x, y)
            fresh.close()
        for x, y in zip([*a.get_state(), a.get_avg_lo()], [*b.get_state(), b.get_avg_lo()]):
            assert torch.equal(x, y), n
        assert a.max_speed() == b.max_speed() and a.counters() == b.counters() and a.status() == b.status()
    a.close()
    b.close()


@pytest.mark.parametrize("asynchronous", [False, True])
def test_upload_equals_load_on_a_large_grid(env, asynchronous):  # noqa: F811
    torch = env[0]
    p = _problem(1025, 609, "inflow")
    st = W.to_f32(W.discretise(p))
    a, b = solver(env, p, state=st), solver(env, p, state=st)
    a.step(0.1 * min(p.dx, p.dy) / a.max_speed())
    (a.set_state_host_async if asynchronous else a.set_state)(*[np.ascontiguousarray(x, dtype=np.float32) for x in st])
    dt = 0.2 * min(p.dx, p.dy) / b.max_speed()
    for _ in range(2):
        assert a.max_speed() == b.max_speed() and a.status() == b.status()
        a.step(dt)
        b.step(dt)
        for x, y in zip([*a.get_state(), a.get_avg_lo()], [*b.get_state(), b.get_avg_lo()]):
            assert torch.equal(x, y)
    a.host_sync()
    a.close()
    b.close()
