"""Values that belong to a wrong place show on data that differ from point to point.
The surrogate's kernel against the sampler's features through the training path's
forward pass, on random data, with the scales that the features give exactly; and
steps whose options change between them, on the untouched tile against every
height that can be set."""
import numpy as np
import pytest

from paper_2508_06273_gb300 import workloads as W
from test_gpu_parity import env, host, solver, to_dev  # noqa: F401
from test_gpu_tile_choice import RIEMANN

pytestmark = pytest.mark.gpu
GAMMA = 1.4


def _random_state(nx, ny, periodic, seed):
    rng = np.random.default_rng(seed)
    out = []
    for k, (w, h) in enumerate(((nx, ny), (nx + 1, ny + 1), (nx + 1, ny), (nx, ny + 1))):
        U = np.stack([rng.uniform(0.8, 1.2, (h, w)), rng.uniform(-0.3, 0.3, (h, w)), rng.uniform(-0.3, 0.3, (h, w)),
                      rng.uniform(0.8, 1.2, (h, w))]).astype(np.float32)
        if k == 0:  # averages: conservative
            E = U[3] / (GAMMA - 1) + 0.5 * U[0] * (U[1] ** 2 + U[2] ** 2)
            U = np.stack([U[0], U[0] * U[1], U[0] * U[2], E])
        elif periodic:
            if w > nx:
                U[:, :, -1] = U[:, :, 0]
            if h > ny:
                U[:, -1] = U[:, 0]
        out.append(np.ascontiguousarray(U, dtype=np.float32))
    return out


@pytest.mark.parametrize("sides", [(0, 0, 0, 0), (1, 1, 1, 1)])
@pytest.mark.parametrize("nx,ny", [(16, 8), (43, 27), (129, 131)])
def test_every_node_gets_its_own_value(env, nx, ny, sides):  # noqa: F811
    torch, af, _ = env
    p = W.fourier_smooth(nx, ny, seed=8, lx=0.1 * nx, ly=0.1 * ny, amp=0.05, modes=2)
    p.bc, p.options = sides, {"ubar": 1}
    st = _random_state(nx, ny, sides[0] == 0, 100 * nx + ny)
    nets = [af.Mlp(seed=s) for s in (3, 4)]
    for n in nets:
        q = n.get_params()
        q[-8:] = 1e-3  # values that stay admissible
        n.set_params(q)
    b = af.Batch([(nx, ny)], [(p.dx, p.dy)], bcs=[p.bc], options=p.options)
    b.set_state(0, *to_dev(torch, st))
    b.set_end(float("inf"), 0.2)
    b.set_sampler(4 * (nx + 1) * (ny + 1), 8 * (nx + 1) * (ny + 1), seed=7, rate=1.0)
    hist = torch.zeros((1, 1), dtype=torch.float64, device="cuda")
    b.run(1, hist)
    Xv, _, idv, Xe, _, ide = b.samples()
    s = solver(env, p, state=st)
    s.set_surrogate(*nets, tol=1e6)
    s.step(float(hist[0, 0]))
    n_net, n_fall = s.surrogate_stats()
    assert n_fall == 0 and n_net == len(Xv) + len(Xe)
    half, new = host(s.get_half()), host(s.get_state())[1:]
    for X, ids, net in ((Xv, idv, nets[0]), (Xe, ide, nets[1])):
        y = net.forward(X).cpu().double().numpy()
        ids, X = ids.cpu().numpy(), X.cpu().double().numpy()
        for kind in np.unique(ids[:, 2]):
            m = ids[:, 2] == kind
            I, J = ids[m, 3] & 0xFFFF, ids[m, 3] >> 16
            U0 = np.asarray(st[1 + kind], dtype=np.float64)[:, J, I]
            # scales rho', c', c', rho' c'^2 from the node's own scaled values: rho = rho' (1 + x),
            # p = rho' c'^2 (1 / gamma + x)
            per, own = (13, 8) if kind == 0 else (15, 9)
            rho = U0[0] / (1 + X[m, own])
            rcc = U0[3] / (1 / GAMMA + X[m, 3 * per + own])
            c = np.sqrt(rcc / rho)
            order = [0, 2, 1, 3] if kind == 2 else [0, 1, 2, 3]
            for lev, got in ((0, half[kind]), (1, new[kind])):
                d = (got[:, J, I] - U0) / np.stack([rho, c, c, rcc])
                want = y[m, 4 * lev:4 * lev + 4].T[order]
                # BF16 activations in both (2^-9 a value in each of three layers, two of them by
                # other GELU roundings) and the FP32 state's step beside values of 1e-3
                tol = 0.1 * np.abs(want).max() + 2e-7
                assert np.abs(d - want).max() < tol, (kind, lev, np.abs(d - want).max(), tol)
                other = np.abs(want - np.roll(want, 1, axis=1)).max(axis=0)  # another row's value is seen
                assert np.mean(other > tol) > 0.9, (kind, lev)
    for x in (b, s, *nets):
        x.close()


@pytest.mark.parametrize("nx,ny", [(33, 21), (129, 121), (130, 300)])
def test_the_tile_follows_the_options(env, nx, ny):  # noqa: F811
    torch = env[0]
    p = W.fourier_smooth(nx, ny, seed=8, lx=0.1 * nx, ly=0.1 * ny, amp=0.05, modes=2)
    state, dt, want = W.to_f32(W.discretise(p)), None, None
    for tile in (None, 4, 8, 16):
        s = solver(env, p, state=state)
        if tile:
            s.set_option("tile_h", tile)
        dt = dt or 0.2 * min(p.dx, p.dy) / s.max_speed()
        got = []
        for options in (RIEMANN, {k: 0 for k in RIEMANN}, {"node_flux": 1}, {"node_flux": 0, "lin_mode": 2}):
            for key, v in options.items():
                s.set_option(key, v)
            s.step(dt)
            s.run(2, dt)
            got += s.get_state()
        want = want or got
        assert all(torch.equal(a, b) for a, b in zip(got, want)), tile
        s.close()
