"""Frames recorded after a state from before the recording's start is loaded: the same steps are
recorded by one call as by single steps (the steps whose distance to the start is a multiple of the
stride, to either side of it)."""
import numpy as np
import pytest

from gpu_helpers import Case, gpu_sim

pytestmark = pytest.mark.gpu


def test_frames_after_loading_an_earlier_state(lblib, tmp_path):
    case = Case(L=8, N=4, steps=0, seed=17)

    def frames(calls):
        sim = gpu_sim(lblib, case, lblib.LB_FP32)
        path = str(tmp_path / "state")
        sim.step(3)
        sim.save(path)
        sim.step(22)
        sim.record_trajectory(stride=10, capacity=16)  # frame 0: step 25
        sim.load(path)                                 # step 3
        for n in calls:
            sim.step(n)
        out = sim.trajectory().cpu().numpy()
        sim.close()
        return out

    one, single = frames([100]), frames([1] * 100)
    assert len(one) == 1 + 10  # steps 5, 15, ..., 95
    assert np.array_equal(one, single)
