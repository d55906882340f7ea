"""Displacements and Rouse correlations on both sides of the rules that choose the staged forms:
short and long chains, few and many lags and modes, runs shorter than the lags, lags that do and do
not fill a block's share.  Against the oracle at 1e-12 of the largest output, as the other sizes
(sums of n terms within a few roundings each, n eps < 1e-12)."""
import numpy as np
import pytest

from oracle import observables as ob

pytestmark = pytest.mark.gpu


def _frames(T, N, seed):
    import torch

    t = np.random.default_rng(seed).normal(size=(T, N, 3)).cumsum(axis=1)
    return t, torch.tensor(t, device="cuda")


def _close(a, b):
    a, b = np.asarray(a), np.asarray(b)
    assert np.max(np.abs(a - b)) <= 1e-12 * max(float(np.max(np.abs(b))), 1e-300)


@pytest.mark.parametrize("T,N,max_lag", [(2, 2100, 1), (9, 500, 20), (7, 600, 9), (41, 120, 3), (400, 22, 60),
                                         (401, 22, 60), (320, 5, 303), (320, 5, 304), (700, 1, 500), (3000, 14, 3)])
def test_displacement_forms(lblib, T, N, max_lag):
    from paper_0903_5067_gb300 import analysis as an

    t, traj = _frames(T, N, T + N)
    for a, b in zip(an.msd(traj, max_lag), ob.msd(t, max_lag)):
        _close(a, b)


@pytest.mark.parametrize("T,P,max_lag", [(70, 75, 10), (70, 76, 10), (9, 80, 130), (33, 38, 63), (33, 38, 64),
                                         (130, 40, 127), (9000, 76, 1), (9001, 76, 1)])
def test_correlation_forms(lblib, T, P, max_lag):
    from paper_0903_5067_gb300 import analysis as an

    X, dev = _frames(T, P, T + P)
    c, x2 = an.rouse_correlation(dev, max_lag)
    co, x2o = ob.rouse_correlation(X, max_lag)
    _close(c, co)
    _close(x2, x2o)
