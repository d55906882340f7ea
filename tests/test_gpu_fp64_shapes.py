"""The FP64 LB kernel over consecutive nodes: boxes on both sides of each block size (one warp to
256 threads), with a last block that is not full and with exactly full ones, with and
without a chain.  FP64 arithmetic against the FP64 oracle: each
population within 1e-12 relative after a few steps, as the FP64 parity tests."""
import numpy as np
import pytest

from gpu_helpers import Case, gpu_sim, oracle_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,N", [(4, 0), (5, 3), (16, 8), (21, 0), (22, 8), (27, 0), (34, 8), (43, 0)])
def test_linear_shapes_match_the_oracle(lblib, L, N):
    case = Case(L=L, N=N, steps=3, seed=40 + L, perturb=0.02)
    st = oracle_run(case)
    sim = gpu_sim(lblib, case, lblib.LB_FP64)
    sim.step(case.steps)
    n = sim.populations()
    assert np.max(np.abs(n - st.n) / np.abs(st.n)) < 1e-12
    if N:
        assert np.max(np.abs(sim.beads()[0] - st.X)) < 1e-12 * L
    sim.close()
