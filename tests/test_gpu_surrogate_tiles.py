"""The fused inference kernel at sizes around its 128-node tiles and on both
sides of the rule that splits the blocks between the two networks: every node's
value against the sampler's features through the training path's forward pass."""
import numpy as np
import pytest

from paper_2508_06273_gb300 import workloads as W
from test_gpu_parity import env, host, solver, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sides", [(0, 0, 0, 0), (1, 1, 1, 1)])
@pytest.mark.parametrize("nx,ny", [(4, 3), (16, 8), (43, 27), (129, 131), (420, 301)])
def test_every_node_gets_its_networks_value(env, nx, ny, sides):  # noqa: F811
    torch, af, _ = env
    p = W.fourier_smooth(nx, ny, seed=8, lx=0.1 * nx, ly=0.1 * ny, amp=0.05, modes=2)
    p.bc = sides
    st = W.to_f32(W.discretise(p))
    nets = [af.Mlp(seed=s) for s in (3, 4)]
    for n in nets:
        q = n.get_params()
        q[-72:-8], q[-8:] = 20.0, 1e-3  # inputs of order one, values that stay admissible
        n.set_params(q)
    b = af.Batch([(nx, ny)], [(p.dx, p.dy)], bcs=[p.bc])
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
    half = host(s.get_half())
    new = host(s.get_state())[1:]
    for X, ids, net in ((Xv, idv, nets[0]), (Xe, ide, nets[1])):
        y = net.forward(X).cpu().double().numpy()
        ids = ids.cpu().numpy()
        X = X.cpu().double().numpy()
        for kind in np.unique(ids[:, 2]):
            m = ids[:, 2] == kind
            I, J = ids[m, 3] & 0xFFFF, ids[m, 3] >> 16
            U0 = np.asarray(st[1 + kind], dtype=np.float64)[:, J, I]
            # scales rho', c', c', rho' c'^2 from the node's primitive data to a few per cent
            c = np.sqrt(1.4 * U0[3] / U0[0])
            scale = np.stack([U0[0], c, c, U0[0] * c * c])
            order = [0, 2, 1, 3] if kind == 2 else [0, 1, 2, 3]
            for lev, got in ((0, half[kind]), (1, new[kind])):
                d = (got[:, J, I] - U0) / scale
                want = y[m, 4 * lev:4 * lev + 4].T[order]
                # bf16 activations (2^-9 each, three layers) and the scales' few per cent
                tol = 0.1 * np.abs(want).max() + 2e-7
                assert np.abs(d - want).max() < tol, (kind, lev, np.abs(d - want).max(), tol)
    for x in (b, s, *nets):
        x.close()
