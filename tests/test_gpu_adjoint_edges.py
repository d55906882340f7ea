"""The adjoint at the edges of its kernels: chains whose entries are ranked and sorted (64 beads fit a
block's threads) and whose scratch fits shared memory or not, and runs of odd and even segments, full
(replayed) and partial.  FP64.

A directional derivative against central differences of the library's own forward run at eps =
1e-5: truncation and cancellation leave about 1e-8 relative there (the adjoint tests), bound 1e-6.
The checkpoint interval changes only where states are recomputed: the same bits."""
import numpy as np
import pytest

from paper_0903_5067_gb300 import inputs

pytestmark = pytest.mark.gpu


def _sim(lb, N, X, zeta=20.8):
    sim = lb.Simulation(L=16, seed=5, precision=lb.LB_FP64)
    sim.add_chain(N, x0=X, zeta=zeta)
    sim._bind()
    return sim


def _objective(lb, N, X, T, zeta=20.8):
    sim = _sim(lb, N, X, zeta)
    sim.step(T)
    x, _ = sim.beads()
    sim.close()
    return float(((x - X) ** 2).sum())


@pytest.mark.parametrize("N", [1, 33, 64, 65, 100])
def test_directional_derivative(lblib, N):
    T, eps = 6, 1e-5
    X = inputs.chain_walk(N, L=16, bond=0.97, seed=60 + N, self_avoiding=True)
    sim = _sim(lblib, N, X)
    _, gx, gz = lblib.lb_adjoint_displacement(sim.ctx, T, 4, N)
    sim.close()
    d = np.random.default_rng(N).normal(size=X.shape)
    fd = (_objective(lblib, N, X + eps * d, T) - _objective(lblib, N, X - eps * d, T)) / (2 * eps)
    assert abs(float((gx * d).sum()) - fd) <= 1e-6 * max(abs(fd), float(np.abs(gx * d).sum()))
    fz = (_objective(lblib, N, X, T, 20.8 + eps) - _objective(lblib, N, X, T, 20.8 - eps)) / (2 * eps)
    assert abs(gz - fz) <= 1e-6 * abs(fz)


@pytest.mark.parametrize("N", [7, 100])
@pytest.mark.parametrize("T,intervals", [(20, (20, 5, 4, 3)), (17, (17, 4, 3, 1))])
def test_checkpoint_intervals(lblib, N, T, intervals):
    X = inputs.chain_walk(N, L=16, bond=0.97, seed=80 + N, self_avoiding=True)
    out = []
    for K in intervals:
        sim = _sim(lblib, N, X)
        O, gx, gz = lblib.lb_adjoint_displacement(sim.ctx, T, K, N)
        x, v = sim.beads()
        sim.step(2)  # the context goes on from the end of the run
        out.append((O, gx, gz, x, v, sim.beads()[0], sim.populations()))
        sim.close()
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert np.array_equal(a, b)
