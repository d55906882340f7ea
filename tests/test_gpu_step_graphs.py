"""Long runs are replayed as CUDA graphs: one call of many steps, single steps, a run cut by samples,
frames and asynchronous read-backs, and a captured call give the same bits."""
import numpy as np
import pytest

from gpu_helpers import Case, gpu_sim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [0, 6])
def test_replayed_steps_equal_single_steps(lblib, N):
    case = Case(L=10, N=N, steps=0, seed=21)

    def state(sim):
        out = [sim.populations()] + (list(sim.beads()) if N else [])
        sim.close()
        return out

    a = gpu_sim(lblib, case, lblib.LB_FP32)
    a.step(131)
    b = gpu_sim(lblib, case, lblib.LB_FP32)
    for _ in range(131):
        b.step(1)
    c = gpu_sim(lblib, case, lblib.LB_FP32)
    c.step(60)
    pops = c.populations()  # applies what is pending: the replay starts from other slots
    c.set_options()         # and the graphs are built again
    c.step(71)
    ref = state(b)
    for sim in (a, c):
        for p, q in zip(state(sim), ref):
            assert np.array_equal(p, q)
    assert pops.shape == ref[0].shape


def test_replayed_steps_with_samples_frames_and_read_backs(lblib):
    import torch

    case = Case(L=10, N=6, steps=0, seed=22)
    a, b = gpu_sim(lblib, case, lblib.LB_FP32), gpu_sim(lblib, case, lblib.LB_FP32)
    x = torch.zeros((2, 18), dtype=torch.float64, pin_memory=True)
    for sim in (a, b):
        lblib.lb_set_obs_stride(sim.ctx, 40)
        sim.record_trajectory(stride=55, capacity=8)
    a.step(90)
    t = lblib.lb_get_beads_async(a.ctx, x[0].numpy(), None, 18)  # the replay rewrites the snapshot it reads
    a.step(130)
    lblib.lb_wait(a.ctx, t)
    for k in range(220):
        b.step(1)
        if k == 89:
            x[1] = torch.from_numpy(b.beads()[0].reshape(-1))
    assert torch.equal(x[0], x[1])
    assert torch.equal(a.trajectory(), b.trajectory()) and a.trajectory().shape[0] == 5
    assert np.array_equal(a.observables(), b.observables()) and a.observables()[17] == 5
    a.close()
    b.close()


def test_captured_steps(lblib):
    """A call on a stream that is being captured records its own launches."""
    import torch

    case = Case(L=10, N=6, steps=0, seed=23)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a, b = gpu_sim(lblib, case, lblib.LB_FP32), gpu_sim(lblib, case, lblib.LB_FP32)
        a.step(50)
        b.step(50)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            a.step(60)
        g.replay()
        b.step(60)
        assert np.array_equal(a.populations(), b.populations())
        assert np.array_equal(a.beads()[0], b.beads()[0])
        a.close()
        b.close()
