"""Rouse correlations by a block per mode and lag and by blocks of lags with the series staged in shared
memory: few lags and many, few modes and many, at the edges of the groups of 32 and 64 lags, against
the oracle at 1e-12 of the largest value as the other observables; and the time of <X_p^2> alone
beside that of 32 lags."""
import numpy as np
import pytest

from oracle import observables as ob

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,P,max_lag", [(60, 3, 0), (40, 90, 0), (40, 90, 3), (40, 90, 31), (40, 90, 32), (70, 16, 63), (70, 16, 64), (70, 2, 68),
                                         (30, 155, 5), (30, 400, 1)])
def test_both_forms(lblib, T, P, max_lag):
    import torch

    from paper_0903_5067_gb300 import analysis as an

    X = np.random.default_rng(T + P).normal(size=(T, P, 3))
    c, x2 = an.rouse_correlation(torch.tensor(X, device="cuda"), max_lag)
    co, x2o = ob.rouse_correlation(X, max_lag)
    assert np.max(np.abs(c - co)) <= 1e-12 * np.max(np.abs(co))
    assert np.max(np.abs(x2 - x2o)) <= 1e-12 * np.max(np.abs(x2o))


def test_one_lag_costs_less_than_32(lblib):
    """The mean squares alone are a thirty-second of the work: they take at most half of the time."""
    import torch

    X = torch.tensor(np.random.default_rng(5).normal(size=(3000, 299, 3)), device="cuda")
    out = torch.empty(299 * 32, dtype=torch.float64, device="cuda")
    s = torch.cuda.current_stream().cuda_stream

    def ms(max_lag):
        best = 1e30
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            for _ in range(20):
                lblib.lb_analysis_rouse_correlation(X.data_ptr(), 3000, 299, max_lag, out.data_ptr(), s)
            e[1].record()
            e[1].synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        return best

    assert ms(0) <= 0.5 * ms(31)
