"""The fluid kernel's rows at the edges of their packing into blocks: rows shorter than a warp, rows
that begin in the middle of a warp, blocks whose last warp or last row group is partly filled, rows
of more than a block, with one node and two nodes per thread, with and without a chain.  Populations
against the FP64 oracle within the FP32 parity bound (1e-5); the largest boxes by their mass, which an
uncovered row of them would change by 1e-5."""
import numpy as np
import pytest

from gpu_helpers import Case, gpu_sim, oracle_run, pop_rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,N", [(4, 0), (5, 0), (18, 0), (31, 0), (36, 0), (40, 0), (51, 16), (58, 16), (72, 16), (82, 0)])
def test_rows_against_the_oracle(lblib, L, N):
    case = Case(L=L, N=N, steps=3, seed=60 + L)
    sim = gpu_sim(lblib, case, lblib.LB_FP32)
    sim.step(case.steps)
    n = sim.populations()
    sim.close()
    assert pop_rel_err(n, oracle_run(case).n) < 1e-5


@pytest.mark.parametrize("L", [257, 300, 514])
def test_large_boxes_keep_their_mass(lblib, L):
    case = Case(L=L, N=0, steps=2, seed=3)
    sim = gpu_sim(lblib, case, lblib.LB_BF16 if L > 500 else lblib.LB_FP32)
    before = sim.observables()
    sim.step(case.steps)
    after = sim.observables()
    sim.close()
    assert abs(after[1] / before[1] - 1.0) < 1e-6
