"""Brownian dynamics at the edges of the kernels' chain lengths (1 to 8 beads per thread, and
the matrix in shared memory beyond), of the Chebyshev degree and of the power iterations, with
and without hydrodynamic interaction, against the FP64 oracle with the bound of the FP32 test:
2e-4 of the largest displacement."""
import numpy as np
import pytest

from oracle import bd
from paper_0903_5067_gb300 import inputs

pytestmark = pytest.mark.gpu


def _walk(N, seed):
    return inputs.chain_walk(N, L=20, bond=0.97, seed=seed, self_avoiding=True)


@pytest.mark.parametrize("N,kw", [(1, {}), (8, {}), (9, dict(hi=False)), (17, dict(degree=1, power_iters=1)),
                                  (24, dict(degree=33)), (32, {}), (33, {}), (41, dict(degree=64)),
                                  (48, {}), (49, {}), (64, {}), (65, {})])
def test_bd_fp32_edges(lblib, N, kw):
    R, steps = 2, 3
    p = bd.BDParams(N=N, seed=6, **kw)
    X0 = np.stack([_walk(N, 20 + N + r) for r in range(R)])
    b = lblib.BD(X0, kT=p.kT, zeta=p.zeta, eta_s=p.eta_s, dt=p.dt, k_fene=p.k_fene, R0=p.R0, eps=p.eps, sigma=p.sigma,
                 hi=p.hi, degree=p.degree, power_iters=p.power_iters, seed=p.seed, precision=lblib.LB_FP32)
    b.step(2)
    b.step(steps - 2)
    x = b.beads()
    b.close()
    for r in range(R):
        ref = bd.run(X0[r], p, steps, replica=r)
        disp = np.abs(ref - X0[r]).max()
        assert np.abs(x[r] - ref).max() <= 2e-4 * disp, r
