"""Free-draining chains of few beads in double precision, where a bead's partners are fewer than the
threads that could share them, against the FP64 oracle with the bound of the FP64 test: 1e-10 of
the largest displacement."""
import numpy as np
import pytest

from oracle import bd
from paper_0903_5067_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 3, 5, 8, 9, 16, 17, 33])
def test_bd_fp64_free_draining(lblib, N):
    p = bd.BDParams(N=N, seed=4, hi=False)
    X0 = np.stack([inputs.chain_walk(N, L=20, bond=0.97, seed=70 + N + r, self_avoiding=True) for r in range(2)])
    b = lblib.BD(X0, kT=p.kT, zeta=p.zeta, eta_s=p.eta_s, dt=p.dt, k_fene=p.k_fene, R0=p.R0, eps=p.eps, sigma=p.sigma,
                 hi=p.hi, seed=p.seed, precision=lblib.LB_FP64)
    b.step(4)
    x = b.beads()
    b.close()
    for r in range(2):
        ref = bd.run(X0[r], p, 4, replica=r)
        assert np.abs(x[r] - ref).max() <= 1e-10 * max(np.abs(ref - X0[r]).max(), 1.0)
