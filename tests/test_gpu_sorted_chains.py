"""Times of chains that need the sorted grouping (more than 128 beads), whose bead step is as long as the
box's whole step, in double precision, beside other times, so that no clock speed enters."""
import numpy as np
import pytest

from paper_0903_5067_gb300 import inputs

pytestmark = pytest.mark.gpu


def _walk(N, seed):
    for again in range(50):
        try:
            return inputs.chain_walk(N, L=24, bond=0.97, seed=seed + 100003 * again, self_avoiding=True)
        except ValueError:
            continue
    raise ValueError("no self-avoiding walk")


def _ms(obj, steps=48):
    """The shortest of five runs of `steps` steps."""
    import torch

    obj.step(steps)
    best = 1e30
    for _ in range(5):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        obj.step(steps)
        e[1].record()
        e[1].synchronize()
        best = min(best, e[0].elapsed_time(e[1]))
    obj.close()
    return best


def _batch(lb, R, N):
    return lb.Batch([24] * R, [N] * R, list(range(R)), [_walk(N, r % 4) for r in range(R)], precision=lb.LB_FP64)


def _box(lb, N):
    sim = lb.Simulation(L=24, precision=lb.LB_FP64, seed=0)
    sim.add_chain(N, x0=_walk(N, 0))
    return sim


@pytest.fixture(scope="module")
def yardstick(lblib):
    """The time of a kernel that is bound by the FP64 pipe as the forces of these chains are: S(k) at 16
    wave numbers of 1000 frames of 128 beads (6.5 ms at 2.07 GHz)."""
    import torch

    traj = torch.tensor(np.random.default_rng(0).normal(size=(1000, 128, 3)).cumsum(axis=1), device="cuda")
    k = torch.tensor([0.1 * 1.25 ** q for q in range(16)], dtype=torch.float64, device="cuda")
    out = torch.empty(16, dtype=torch.float64, device="cuda")
    best = 1e30
    for _ in range(6):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        lblib.lb_analysis_static_sk(traj.data_ptr(), 1000, 128, k.data_ptr(), 16, out.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream)
        e[1].record()
        e[1].synchronize()
        best = min(best, e[0].elapsed_time(e[1]))
    return best


def test_batch(lblib, yardstick):
    """0.68 ms per step at 2.07 GHz; with the marks of the nodes set in a loop 0.75."""
    assert _ms(_batch(lblib, 1, 200)) / 48 <= 0.110 * yardstick


def test_box(lblib, yardstick):
    """0.61 ms per step at 2.07 GHz on blocks of 512 threads; 0.68 on 256."""
    assert _ms(_box(lblib, 200)) / 48 <= 0.099 * yardstick


def test_as_many_chains_as_there_is_room_for(lblib):
    """A block per chain and many more SMs than chains: 32 take no longer than 2 (5 % are allowed)."""
    assert _ms(_batch(lblib, 32, 200)) <= 1.05 * _ms(_batch(lblib, 2, 200))
