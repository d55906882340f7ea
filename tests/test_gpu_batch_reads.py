"""Reading a replica's observables and populations waits for the device once: they do not report the
device status, which a box's do at the price of another copy and wait."""
import time

import numpy as np
import pytest

from paper_0903_5067_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_a_replica_is_read_faster_than_a_box(lblib):
    """The same observables of the same L = 16: 43 us of a replica, 49 of a box; 50 with the status."""
    x = inputs.chain_walk(8, L=16, bond=0.97, seed=3, self_avoiding=True)
    sim = lblib.Simulation(L=16, precision=lblib.LB_FP32, seed=5)
    sim.add_chain(8, x0=x)
    b = lblib.Batch([16], [8], [5], [x], precision=lblib.LB_FP32)
    for obj in (sim, b):
        obj.step(2)

    def us(call):
        times = []
        for _ in range(200):
            t = time.perf_counter()
            call()
            times.append(time.perf_counter() - t)
        return 1e6 * min(times)

    assert np.array_equal(b.observables(0), sim.observables()) and np.array_equal(b.populations(0), sim.populations())
    assert us(lambda: b.observables(0)) <= 0.955 * us(sim.observables)
    sim.close()
    b.close()
