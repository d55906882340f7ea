"""The bead step at the edges of its splits: chains that do not fill a block or a cluster evenly,
the largest chain and substep counts grouped by cells and the smallest that are sorted, boxes so
small that every cell touches its own images' neighbours, lattice spacings and masses whose
reciprocals are not exact, and replicas of a batch on every cluster size beside chains that are
sorted and boxes without one.  Against the FP64 oracle, with the bounds of the parity tests: FP64
1e-12 per population and of the box per bead coordinate, FP32 1e-5 and 1e-6."""
import numpy as np
import pytest

from gpu_helpers import Case, gpu_sim, oracle_run, pop_rel_err
from oracle import lbchain as o
from paper_0903_5067_gb300 import inputs

pytestmark = pytest.mark.gpu

EDGES = [
    Case(L=4, N=3, steps=4, seed=2),
    Case(L=5, N=9, steps=4, seed=3, ext=(0.3, -0.2, 0.1), counter=True),
    Case(L=7, N=2, steps=5, seed=4, a=0.8, m=1.3, h=0.02),
    Case(L=9, N=17, steps=4, seed=5, substeps=2),
    Case(L=12, N=33, steps=3, seed=6, a=1.1),
    Case(L=14, N=64, steps=2, seed=7, substeps=2),   # 1024 corners: the most compared
    Case(L=14, N=43, steps=2, seed=8, substeps=3),   # 1032: sorted
    Case(L=20, N=128, steps=2, seed=9),
    Case(L=20, N=129, steps=2, seed=10),
]


def _check(n, x, st, L, a, prec_fp64):
    assert pop_rel_err(n, st.n) < (1e-12 if prec_fp64 else 1e-5)
    if x is not None:
        assert np.max(np.abs(x - st.X)) < (1e-12 if prec_fp64 else 1e-6) * L * a


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("case", EDGES, ids=lambda c: f"L{c.L}-N{c.N}-s{c.substeps}")
def test_bead_step_edges(lblib, case, prec):
    if prec == "fp32" and case.h > 0.01:
        pytest.skip("the FP32 bound is the parity tests', at their noise amplitude (h = 0.01, a = 1)")
    sim = gpu_sim(lblib, case, lblib.LB_FP64 if prec == "fp64" else lblib.LB_FP32)
    sim.step(case.steps)
    n, (x, _) = sim.populations(), sim.beads()
    sim.close()
    _check(n, x, oracle_run(case), case.L, case.a, prec == "fp64")


@pytest.mark.parametrize("R,sub", [(2, 1), (19, 2), (50, 1), (160, 1)])
def test_batch_cluster_sizes(lblib, R, sub):
    N = [(12, 0, 5, 33)[r % 4] for r in range(R)]
    if R == 2:
        N = [140, 7]  # a sorted chain beside one on a cluster
    L = [(8, 5, 9, 12)[r % 4] for r in range(R)]
    if R == 2:
        L = [20, 6]
    seeds = [200 + r for r in range(R)]
    X = [inputs.chain_walk(n, L=l, bond=0.97, seed=s, self_avoiding=True) for n, l, s in zip(N, L, seeds)]
    b = lblib.Batch(L, N, seeds, X, precision=lblib.LB_FP64, md_substeps=sub)
    b.step(3)
    for r in {0, 1, R // 2, R - 1}:
        fp = o.FluidParams(L=L[r], rho=1.0, eta=3.0, eta_b=3.0, kT=1.0, h=0.01, a=1.0, seed=seeds[r])
        cp = o.ChainParams(N=N[r], substeps=sub) if N[r] else None
        st = o.run(o.init_state(fp, cp, X[r] if cp else None), fp, cp, 3, replica=r)
        _check(b.populations(r), b.beads(r)[0] if cp else None, st, L[r], 1.0, True)
    b.close()
