"""Trajectories with a position that is not a number: what depends on it is not a number either, in the
oracle and in the kernels, and everything else keeps its value (1e-12 of the largest finite one,
as for finite trajectories)."""
import numpy as np
import pytest

from oracle import observables as ob

pytestmark = pytest.mark.gpu


def _frames(T, N, seed, where):
    import torch

    t = np.random.default_rng(seed).normal(size=(T, N, 3)).cumsum(axis=1)
    t[where] = np.nan
    return t, torch.tensor(t, device="cuda")


def _same(a, b):
    a, b = np.asarray(a), np.asarray(b)
    ok = np.isfinite(b)
    assert np.array_equal(np.isfinite(a), ok)
    assert np.max(np.abs(a[ok] - b[ok]), initial=0.0) <= 1e-12 * np.max(np.abs(b[ok]), initial=1e-300)


@pytest.mark.parametrize("N", [3, 8, 17])
@pytest.mark.parametrize("place", ["first", "middle", "last"])
def test_rouse_modes(lblib, N, place):
    from paper_0903_5067_gb300 import analysis as an

    n = {"first": 0, "middle": N // 2, "last": N - 1}[place]
    t, traj = _frames(6, N, N, (2, n, 1))
    _same(an.rouse_modes(traj).cpu().numpy(), ob.rouse_modes(t))


@pytest.mark.parametrize("ks", [[0.0], [0.0, 0.7, 1.3], [0.9, 1.1]])
def test_structure_factors(lblib, ks):
    from paper_0903_5067_gb300 import analysis as an

    t, traj = _frames(4, 5, 11, (3, 1, 2))
    _same(an.static_sk(traj, ks), ob.static_structure_factor(t, ks))
    _same(an.dynamic_sk(traj, ks, 3, origin_stride=3), ob.dynamic_structure_factor(t, ks, 3, origin_stride=3))
    assert np.isnan(an.inverse_radius(traj))
