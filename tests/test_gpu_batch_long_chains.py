"""Batches of chains that need more than one block each: beside other replicas than blocks have SMs, in
large boxes, and mixed with short chains and none.  Against the FP64 oracle, with the FP32 bounds of
the parity tests: 1e-5 per population and 1e-6 of the box per bead coordinate.  And the step of large
boxes takes no longer for a long chain, whose bead kernel runs beside the fluid's."""
import numpy as np
import pytest

from gpu_helpers import pop_rel_err
from oracle import lbchain as o
from paper_0903_5067_gb300 import inputs

pytestmark = pytest.mark.gpu


def _walk(N, L, seed):
    for again in range(50):
        try:
            return inputs.chain_walk(N, L=L, bond=0.97, seed=seed + 100003 * again, self_avoiding=True)
        except ValueError:
            continue
    raise ValueError("no self-avoiding walk")


@pytest.mark.parametrize("R,L,N,sub,large", [(80, 10, (65, 3, 0), 1, 0), (160, 9, (33, 0, 40), 2, 0), (3, 12, (128, 9, 5), 1, 0),
                                             (3, 14, (128, 1, 70), 1, 128), (2, 11, (64, 20, 2), 2, 130)])
def test_against_the_oracle(lblib, R, L, N, sub, large):
    """`large`: one more box of that size, for a batch whose fluid sets the step."""
    Ls, Ns = [L] * R + [large] * (large > 0), [N[r % 3] for r in range(R)] + [N[0]] * (large > 0)
    seeds = [700 + r for r in range(len(Ls))]
    X = [_walk(n, l, s) for n, l, s in zip(Ns, Ls, seeds)]
    b = lblib.Batch(Ls, Ns, seeds, X, precision=lblib.LB_FP32, md_substeps=sub)
    b.step(3)
    for r in {0, 1, 2 % R, R - 1}:
        fp = o.FluidParams(L=Ls[r], rho=1.0, eta=3.0, eta_b=3.0, kT=1.0, h=0.01, a=1.0, seed=seeds[r])
        cp = o.ChainParams(N=Ns[r], substeps=sub) if Ns[r] else None
        st = o.run(o.init_state(fp, cp, X[r] if cp else None), fp, cp, 3, replica=r)
        assert pop_rel_err(b.populations(r), st.n) < 1e-5
        if cp:
            assert np.max(np.abs(b.beads(r)[0] - st.X)) < 1e-6 * Ls[r]
    b.close()


def test_a_long_chain_hides_behind_the_fluid(lblib):
    """Three boxes of L = 100: 70 us per step of the fluid; a chain of 128 beads may add a quarter to what
    one of 8 takes."""
    import torch

    def ms(N):
        b = lblib.Batch([100] * 3, [N] * 3, [1, 2, 3], [_walk(N, 100, s) for s in (1, 2, 3)], precision=lblib.LB_FP32)
        b.step(32)
        best = 1e30
        for _ in range(5):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            b.step(64)
            e[1].record()
            e[1].synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        b.close()
        return best

    assert ms(128) <= 1.25 * ms(8)
