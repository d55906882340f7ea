"""The double-precision noise tables are one per device: contexts that start at the same time on
several threads and streams, and contexts after all earlier ones are gone, give the same states bit
for bit."""
import threading

import numpy as np
import pytest

from gpu_helpers import Case, gpu_sim

pytestmark = pytest.mark.gpu


def test_contexts_started_together(lblib):
    import torch

    case = Case(L=9, N=5, steps=6, seed=12)

    def run(out, k):
        with torch.cuda.stream(torch.cuda.Stream()):
            sim = gpu_sim(lblib, case, lblib.LB_FP64)
            sim.step(case.steps)
            out[k] = (sim.populations(), sim.beads()[0])
            sim.close()

    out = {}
    threads = [threading.Thread(target=run, args=(out, k)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    run(out, 4)
    for k in range(1, 5):
        assert np.array_equal(out[k][0], out[0][0]) and np.array_equal(out[k][1], out[0][1])
