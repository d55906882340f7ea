"""One step of a perturbed fluid in boxes whose rows take more than one block of the fluid kernel, and at
the edge between the double-precision kernel over consecutive nodes (L <= 256) and the one over rows,
against the oracle's single-node update at sampled nodes: the first and last places of each row
segment, rows and planes, whose pull sources wrap around, and random ones.  Bounds as in the parity
tests: 1e-12 and 1e-5 per population in FP64 and FP32; in BF16 8 roundings of the largest deviation.
With a chain the total momentum, which the coupled step conserves: to 1e-13 of a momentum of one per node
(2e-4, far above the rounding of L^3 nodes in FP64; a bead's impulse, which a correction left out would take
away, is of the order of 0.1)."""
import numpy as np
import pytest

from oracle import lbchain as o

pytestmark = pytest.mark.gpu


def _h(i, z, y, x):
    """A field of -1 ... 1 in steps of 1/128 that no shift of a coordinate leaves as it is; for integers and
    integer tensors."""
    return ((3 * x * x + 5 * y * y + 7 * z * z + x * y + 13 * y * z + 11 * i * x + 17 * i) % 257) / 128.0 - 1.0


class _Field:
    """The initial populations as the oracle's node update indexes them."""

    def __init__(self, rest):
        self.rest = rest  # w_i rho

    def __getitem__(self, at):
        i, z, y, x = (int(v) for v in at)
        return self.rest[i] * (1.0 + 0.03125 * _h(i, z, y, x))


def _fill(out, L, rest):
    import torch

    c = torch.arange(L, device="cuda")
    for i in range(19):
        h = _h(i, c[:, None, None], c[None, :, None], c[None, None, :])
        out[i].copy_(rest[i] * (1.0 + 0.03125 * h.double()))


def _nodes(L):
    rng = np.random.default_rng(L)
    edge = sorted({0, 1, 127, 128, 255, min(256, L - 1), L // 2, L - 2, L - 1})
    nodes = {(x, y, z) for x in edge for y in (0, 1, 255, L - 1) for z in (0, 128, L - 1)}
    nodes |= {(L // 3, y, z) for y in edge for z in edge}
    return sorted(nodes | {tuple(int(c) for c in rng.integers(0, L, 3)) for _ in range(200)})


@pytest.mark.parametrize("L,N,precision", [(256, 0, "FP64"), (257, 0, "FP64"), (256, 5, "FP64"), (257, 5, "FP64"), (257, 0, "FP32"),
                                           (300, 0, "FP32"), (257, 5, "FP32"), (300, 5, "FP32"), (514, 0, "BF16")])
def test_sampled_nodes_after_one_step(lblib, L, N, precision):
    import torch

    fp = o.FluidParams(L=L, rho=1.0, eta=3.0, eta_b=3.0, kT=1.0, h=0.01, a=1.0, seed=9)
    rest = [float(w) * fp.rho for w in [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12]
    buf = torch.empty((19, L, L, L), dtype=torch.float64, pin_memory=True)
    _fill(buf, L, rest)
    torch.cuda.synchronize()
    n = buf.numpy()
    sim = lblib.Simulation(L=L, rho=fp.rho, eta=fp.eta, eta_b=fp.eta_b, kT=fp.kT, h=fp.h, a=fp.a, seed=fp.seed,
                           precision=getattr(lblib, "LB_" + precision))
    if N:  # in a corner of the box, away from the sampled edges' rows
        sim.add_chain(N, x0=np.array([[40.3 + 0.9 * b, 71.6, 33.2] for b in range(N)]))
    sim.set_populations(n)
    sim._bind()
    before = sim.observables()[2:5]
    sim.step(1)
    lblib.lb_get_populations(sim.ctx, n)
    field, worst, dev = _Field(rest), 0.0, 0.0
    for x, y, z in _nodes(L):
        if N and abs(x - 42) < 6 and abs(y - 71) < 4 and abs(z - 33) < 4:
            continue
        want = o.node_update(field, fp, 0, (x, y, z))
        got = n[:, z, y, x]
        dev = max(dev, float(np.max(np.abs(want - rest))))
        worst = max(worst, float(np.max(np.abs(got - want) / (1.0 if precision == "BF16" else np.abs(want)))))
    assert worst <= {"FP64": 1e-12, "FP32": 1e-5, "BF16": 8 * 2.0 ** -8 * dev}[precision]
    if N and precision == "FP64":
        sim.step(3)
        after = sim.observables()[2:5]
        assert np.all(np.abs(after - before) <= 1e-13 * L ** 3 * fp.a / fp.h)
    sim.close()
