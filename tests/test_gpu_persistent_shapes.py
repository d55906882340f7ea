"""Batches on persistent blocks of the fluid kernel: the same states as on one block per tile, bit for bit,
with chains of one and of two bead blocks and without; and their time beside that."""
import numpy as np
import pytest

from paper_0903_5067_gb300 import inputs

pytestmark = pytest.mark.gpu


def _walk(N, L, seed):
    for again in range(50):
        try:
            return inputs.chain_walk(N, L=L, bond=0.97, seed=seed + 100003 * again, self_avoiding=True)
        except ValueError:
            continue
    raise ValueError("no self-avoiding walk")


def _batch(lb, L, N, precision, shape):
    b = lb.Batch(L, N, list(range(len(L))), [_walk(n, l, r % 4) for r, (l, n) in enumerate(zip(L, N))], precision=precision)
    lb.lb_batch_set_shape(b.b, *shape)
    return b


@pytest.mark.parametrize("precision", ["LB_FP32", "LB_FP64"])
@pytest.mark.parametrize("shape", [(128, 1), (256, 2), (512, 4)])
def test_the_same_states(lblib, precision, shape):
    L, N = [16, 11, 12, 9, 16, 7], [30, 0, 70, 5, 100, 2]
    states = []
    for s in ((256, 0), shape):
        b = _batch(lblib, L, N, getattr(lblib, precision), s)
        b.step(21)
        states.append([b.populations(r) for r in range(len(L))] + [b.beads(r)[0] for r in range(len(L)) if N[r]])
        b.close()
    assert all(np.array_equal(a, c) for a, c in zip(*states))


def test_time(lblib):
    """One block of 128 threads per SM takes 3.1 times what a block per tile takes (64 replicas of L = 32);
    3.3 with registers spilled in its loop."""
    import torch

    def ms(shape):
        b = _batch(lblib, [32] * 64, [16] * 64, lblib.LB_FP32, shape)
        b.step(32)
        best = 1e30
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            b.step(48)
            e[1].record()
            e[1].synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        b.close()
        return best

    assert ms((128, 1)) <= 3.18 * ms((128, 0))
