"""The forms of the structure factors and the hydrodynamic radius: by a block without a table of sines, by
one cluster and by two per group of wave numbers, on frames of fewer pairs than threads and of more,
against the oracle at 1e-12 of the largest value as the other observables; and the time of many
frames of few pairs beside few frames of many."""
import numpy as np
import pytest

from oracle import observables as ob

pytestmark = pytest.mark.gpu


def _frames(T, N, seed):
    import torch

    t = np.random.default_rng(seed).normal(size=(T, N, 3)).cumsum(axis=1)
    return t, torch.tensor(t, device="cuda")


def _close(a, b):
    assert np.max(np.abs(np.asarray(a) - np.asarray(b))) <= 1e-12 * np.max(np.abs(b))


@pytest.mark.parametrize("T,N,nk", [(1, 1, 2), (255, 2, 1), (257, 2, 3), (700, 2, 2), (90, 4, 1), (60, 9, 4), (35, 23, 1),
                                    (8, 24, 16), (9, 33, 5), (2, 70, 9), (3, 91, 2)])
def test_static(lblib, T, N, nk):
    from paper_0903_5067_gb300 import analysis as an

    t, traj = _frames(T, N, T + 1000 * N)
    ks = [0.0 if q == 1 else 0.1 * 1.4 ** q for q in range(nk)]
    _close(an.static_sk(traj, ks), ob.static_structure_factor(t, ks))
    if N > 1:
        assert an.inverse_radius(traj) == pytest.approx(ob.inverse_hydrodynamic_radius(t), rel=1e-12)


@pytest.mark.parametrize("T,N,nk,lag,stride", [(300, 2, 1, 3, 1), (90, 2, 16, 2, 1), (40, 3, 4, 12, 7), (9, 13, 16, 1, 1), (12, 16, 2, 3, 3),
                                               (20, 12, 3, 1, 1), (4, 33, 5, 1, 1), (3, 46, 2, 4, 2), (2, 65, 4, 1, 1)])
def test_dynamic(lblib, T, N, nk, lag, stride):
    from paper_0903_5067_gb300 import analysis as an

    t, traj = _frames(T, N, T + 1000 * N)
    ks = [0.1 * 1.4 ** q for q in range(nk)]
    _close(an.dynamic_sk(traj, ks, lag, origin_stride=stride), ob.dynamic_structure_factor(t, ks, lag, origin_stride=stride))


def test_many_short_frames_take_as_long_as_few_long_ones(lblib):
    """8128 pairs in 8128 frames of 2 beads and in one of 128: the same sums.  Twice the time is allowed (for
    S(k) without the pairs of a bead with itself, for S(k, t) with them: 16384 against 16384)."""
    import torch

    k = torch.tensor([0.1 * 1.2 ** q for q in range(16)], dtype=torch.float64, device="cuda")
    out = torch.empty(64, dtype=torch.float64, device="cuda")
    s = torch.cuda.current_stream().cuda_stream

    def us(call):
        best = 1e30
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            for _ in range(20):
                call()
            e[1].record()
            e[1].synchronize()
            best = min(best, e[0].elapsed_time(e[1]) * 50)
        return best

    _, short = _frames(8128, 2, 1)
    _, long = _frames(1, 128, 1)
    _, short4 = _frames(4096, 2, 1)
    p = [x.data_ptr() for x in (short, long, short4, k, out)]
    for many, few in (
            (lambda: lblib.lb_analysis_static_sk(p[0], 8128, 2, p[3], 16, p[4], s),
             lambda: lblib.lb_analysis_static_sk(p[1], 1, 128, p[3], 16, p[4], s)),
            (lambda: lblib.lb_analysis_dynamic_sk(p[2], 4096, 2, p[3], 16, 0, 1, p[4], s),
             lambda: lblib.lb_analysis_dynamic_sk(p[1], 1, 128, p[3], 16, 0, 1, p[4], s)),
            (lambda: lblib.lb_analysis_inverse_radius(p[0], 8128, 2, p[4], s),
             lambda: lblib.lb_analysis_inverse_radius(p[1], 1, 128, p[4], s))):
        assert us(many) <= 2.0 * us(few)
