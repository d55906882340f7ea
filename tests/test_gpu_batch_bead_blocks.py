"""Single-precision batches on both sizes of the bead step's blocks: few corners per block, and more
than 96 (12 beads per block of 40 replicas with two substeps, all 33 beads of 160 replicas), beside
boxes without a chain.  Against the FP64 oracle, with the FP32 bounds of the parity tests: 1e-5 per
population and 1e-6 of the box per bead coordinate."""
import numpy as np
import pytest

from gpu_helpers import pop_rel_err
from oracle import lbchain as o
from paper_0903_5067_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,sub", [(3, 1), (40, 2), (160, 1)])
def test_batch_bead_blocks(lblib, R, sub):
    N = [(33, 0, 12, 2)[r % 4] for r in range(R)]
    L = [(11, 5, 9, 6)[r % 4] for r in range(R)]
    seeds = [300 + r for r in range(R)]
    X = [inputs.chain_walk(n, L=l, bond=0.97, seed=s, self_avoiding=True) for n, l, s in zip(N, L, seeds)]
    b = lblib.Batch(L, N, seeds, X, precision=lblib.LB_FP32, md_substeps=sub)
    b.step(3)
    for r in {0, 1, R // 2, R - 1}:
        fp = o.FluidParams(L=L[r], rho=1.0, eta=3.0, eta_b=3.0, kT=1.0, h=0.01, a=1.0, seed=seeds[r])
        cp = o.ChainParams(N=N[r], substeps=sub) if N[r] else None
        st = o.run(o.init_state(fp, cp, X[r] if cp else None), fp, cp, 3, replica=r)
        assert pop_rel_err(b.populations(r), st.n) < 1e-5
        if cp:
            assert np.max(np.abs(b.beads(r)[0] - st.X)) < 1e-6 * L[r]
    b.close()
