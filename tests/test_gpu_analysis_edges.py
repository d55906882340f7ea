"""Edges of the chain-observable kernels against the oracle: odd and even chains, pairs and
origins that do not fill a block or a cluster, coincident and near-coincident beads, wave
numbers of both argument ranges (and 0), every group size of wave numbers, and both sides of
the run lengths that are staged in shared memory.

Tolerance: every output is a sum of n terms each within a few roundings of its exact value,
compared at 1e-12 of the largest output as the other observables are (n eps < 1e-12 for the
sizes here)."""
import numpy as np
import pytest

from oracle import observables as ob

pytestmark = pytest.mark.gpu


def _close(a, b, rtol=1e-12):
    a, b = np.asarray(a), np.asarray(b)
    scale = max(float(np.max(np.abs(b))), 1e-300)
    assert np.max(np.abs(a - b)) <= rtol * scale, (np.max(np.abs(a - b)), scale)


def _frames(T, N, seed):
    import torch

    t = np.random.default_rng(seed).normal(size=(T, N, 3)).cumsum(axis=1)
    return t, torch.tensor(t, device="cuda")


@pytest.mark.parametrize("T,N,nk", [(1, 2, 1), (2, 3, 2), (5, 17, 3), (3, 32, 4), (2, 33, 5), (1, 40, 8), (2, 21, 9),
                                    (1, 24, 17)])
def test_structure_factors_and_radius(lblib, T, N, nk):
    from paper_0903_5067_gb300 import analysis as an

    t, traj = _frames(T, N, 100 * N + T)
    ks = [0.05 * 1.7 ** q for q in range(nk)]
    _close(an.static_sk(traj, ks), ob.static_structure_factor(t, ks))
    _close(an.dynamic_sk(traj, ks, T, origin_stride=2), ob.dynamic_structure_factor(t, ks, T, origin_stride=2))
    assert an.inverse_radius(traj) == pytest.approx(ob.inverse_hydrodynamic_radius(t), rel=1e-12)


def test_structure_factor_general_arguments(lblib):
    """Coincident beads (sinc = 1), distances whose square leaves the range of the fast 1/r, k = 0
    and arguments past the table's range, alone and beside ordinary ones."""
    from paper_0903_5067_gb300 import analysis as an

    import torch

    t, _ = _frames(2, 6, 7)
    t[:, 1] = t[:, 0]
    t[:, 2] = t[:, 0] + 1e-20
    t[0, 5] = 1e18
    traj = torch.tensor(t, device="cuda")
    for ks in ([0.0], [0.7, 0.0, 1.1], [1e-3, 3e6], [0.0] * 5 + [0.9] * 5):
        _close(an.static_sk(traj, ks), ob.static_structure_factor(t, ks))
        _close(an.dynamic_sk(traj, ks, 1), ob.dynamic_structure_factor(t, ks, 1))
    t[:, 1:3] += [[0.1, 0, 0], [1e-17, 3, 0]]
    assert an.inverse_radius(torch.tensor(t, device="cuda")) == pytest.approx(ob.inverse_hydrodynamic_radius(t),
                                                                              rel=1e-12)


@pytest.mark.parametrize("T,N,max_lag", [(1, 1, 0), (7, 2, 9), (9, 95, 3), (40, 97, 12), (3000, 3, 2), (3001, 3, 2)])
def test_displacements(lblib, T, N, max_lag):
    from paper_0903_5067_gb300 import analysis as an

    t, traj = _frames(T, N, 31 * T + N)
    for a, b in zip(an.msd(traj, max_lag), ob.msd(t, max_lag)):
        _close(a, b)


@pytest.mark.parametrize("T,N,P", [(1, 2, 1), (3, 3, 2), (5, 16, 15), (4, 33, 32), (6, 128, 100), (9, 1700, 3)])
def test_rouse_modes(lblib, T, N, P):
    from paper_0903_5067_gb300 import analysis as an

    t, traj = _frames(T, N, 7 * T + N)
    _close(an.rouse_modes(traj, P).cpu().numpy(), ob.rouse_modes(t, P))


@pytest.mark.parametrize("T,P,max_lag", [(1, 1, 0), (5, 2, 8), (150, 2, 141), (9000, 1, 1), (9001, 1, 1)])
def test_rouse_correlation(lblib, T, P, max_lag):
    from paper_0903_5067_gb300 import analysis as an

    X, dev = _frames(T, P, 3 * T + P)
    c, x2 = an.rouse_correlation(dev, max_lag)
    co, x2o = ob.rouse_correlation(X, max_lag)
    _close(c, co)
    _close(x2, x2o)
