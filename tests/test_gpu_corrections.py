"""The force corrections that the fluid kernels add by warp, where the sharing out can go wrong: a
straight chain along a row, which marks all 64 nodes of a warp with two nodes per thread (two
passes of 32), rows whose last warp holds one node or pair, FP64 boxes whose last warp is partly
filled, and chains across the periodic faces.  Against the FP64 oracle, with the bounds of the parity
tests: FP64 1e-12 per population and of the box per bead coordinate, FP32 1e-5 and 1e-6."""
import dataclasses

import numpy as np
import pytest

from gpu_helpers import Case, gpu_sim, oracle_run, pop_rel_err
from oracle import lbchain as o

pytestmark = pytest.mark.gpu


@dataclasses.dataclass(frozen=True)
class RowCase(Case):
    """A straight chain along x, off the lattice points along y and z."""

    start: tuple = (1.3, 2.4, 3.6)

    def x0(self):
        return np.array(self.start) + 0.97 * np.arange(self.N)[:, None] * np.array([1.0, 0.0, 0.0])


ROWS = [
    RowCase(L=64, N=62, steps=3, seed=31),                           # two full passes
    RowCase(L=66, N=64, steps=2, seed=32, start=(0.2, 65.7, 65.9)),  # rows of 33 pairs, across two faces
    RowCase(L=33, N=31, steps=3, seed=33, start=(1.3, 32.5, 0.5)),   # rows of a warp and one node
    RowCase(L=9, N=7, steps=4, seed=34, start=(0.5, 8.5, 8.5)),      # 729 nodes
    RowCase(L=8, N=6, steps=4, seed=35, substeps=2),                 # rows of four pairs
]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("case", ROWS, ids=lambda c: f"L{c.L}")
def test_row_of_marked_nodes(lblib, case, prec):
    sim = gpu_sim(lblib, case, lblib.LB_FP64 if prec == "fp64" else lblib.LB_FP32)
    sim.step(case.steps)
    n, (x, _) = sim.populations(), sim.beads()
    sim.close()
    st = oracle_run(case)
    assert pop_rel_err(n, st.n) < (1e-12 if prec == "fp64" else 1e-5)
    assert np.max(np.abs(x - st.X)) < (1e-12 if prec == "fp64" else 1e-6) * case.L


@pytest.mark.parametrize("shape", [(256, 0), (512, 2)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_batched_rows(lblib, prec, shape):
    """Replicas of both tile forms side by side, by one block per tile and by persistent blocks."""
    cases = [ROWS[0], ROWS[2], ROWS[3], ROWS[0]]
    cases = [dataclasses.replace(c, steps=3, seed=40 + r, substeps=1) for r, c in enumerate(cases)]
    b = lblib.Batch([c.L for c in cases], [c.N for c in cases], [c.seed for c in cases], [c.x0() for c in cases],
                    precision=lblib.LB_FP64 if prec == "fp64" else lblib.LB_FP32)
    lblib.lb_batch_set_shape(b.b, *shape)
    b.step(3)
    for r, c in enumerate(cases):
        fp, cp = c.fluid(), c.chain()
        st = o.run(o.init_state(fp, cp, c.x0()), fp, cp, 3, replica=r)
        assert pop_rel_err(b.populations(r), st.n) < (1e-12 if prec == "fp64" else 1e-5)
        assert np.max(np.abs(b.beads(r)[0] - st.X)) < (1e-12 if prec == "fp64" else 1e-6) * c.L
    b.close()
