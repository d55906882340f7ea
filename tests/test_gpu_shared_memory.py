"""Objects and calls whose kernels need different amounts of shared memory beyond the 48 KB that need
no asking, side by side: the largest made first and used last, calls from two threads at once, and a
batch whose bead kernel passes 48 KB only together with its static part.  Nothing is refused, and
the results are those of each alone."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _grid_chain(N, at):
    """A chain that winds through a lattice of 16 x 8 x 8 places from the point `at` on: bonds of 0.97 along
    the rows of 16 and 1.15 between them, no two other beads closer than 1.15."""
    i = np.arange(N)
    x, y, z = i % 16, i // 16 % 8, i // 128
    x = np.where((i // 16) % 2, 15 - x, x)
    y = np.where(z % 2, 7 - y, y)
    return np.stack([0.97 * x, 1.15 * y, 1.15 * z], axis=1) + at


def _batch(lb, N, substeps, precision, L=20, R=80):
    return lb.Batch([L] * R, [N] * R, list(range(R)), [_grid_chain(N, 1.3 + 0.001 * r) for r in range(R)],
                    precision=precision, md_substeps=substeps)


def _box(lb, N, precision):
    sim = lb.Simulation(L=20, precision=precision)
    sim.add_chain(N, x0=_grid_chain(N, 1.3))
    return sim


def _bd(lb, N, precision):
    return lb.BD(np.stack([_grid_chain(N, 0.0)] * 2), precision=precision)


def _objects(lb, kind, precision):
    """[(make, steps)] of objects in order of decreasing need."""
    prec = getattr(lb, precision)
    if kind == "batch":  # one block per chain
        return [lambda: _batch(lb, 64, 2, prec), lambda: _batch(lb, 48, 2, prec), lambda: _batch(lb, 76, 1, prec)]
    if kind == "box":  # the sorted bead step
        return [lambda: _box(lb, 1000, prec), lambda: _box(lb, 600, prec)]
    return [lambda: _bd(lb, 52, prec), lambda: _bd(lb, 45, prec), lambda: _bd(lb, 33, prec)] if precision == "LB_FP64" else \
        [lambda: _bd(lb, 74, prec), lambda: _bd(lb, 66, prec), lambda: _bd(lb, 64, prec), lambda: _bd(lb, 50, prec)]


def _state(obj):
    return obj.beads(0)[0] if hasattr(obj, "L") and isinstance(obj.L, list) else \
        (obj.beads()[0] if hasattr(obj, "L") else obj.beads())


@pytest.mark.parametrize("precision", ["LB_FP32", "LB_FP64"])
@pytest.mark.parametrize("kind", ["batch", "box", "bd"])
def test_the_largest_first_and_last(lblib, kind, precision):
    makes = _objects(lblib, kind, precision)
    alone = []
    for make in reversed(makes):  # the smallest first: nothing before it asked for more
        obj = make()
        obj.step(3)
        alone.append(_state(obj))
        obj.close()
    objs = [make() for make in makes]
    for obj in objs:
        obj.step(0)  # on the device
    for obj in reversed(objs):
        obj.step(3)
    for obj, want in zip(objs, reversed(alone)):
        assert np.array_equal(_state(obj), want)
        obj.close()


def test_adjoints_of_long_and_short_chains(lblib):
    def grad(N):
        sim = _box(lblib, N, lblib.LB_FP32)
        sim._bind()
        out = lblib.lb_adjoint_displacement(sim.ctx, 3, 3, N)
        sim.close()
        return out

    first, _, again = grad(64), grad(40), grad(64)
    assert np.array_equal(first[1], again[1])


def test_observables_from_two_threads(lblib):
    """Displacements, Rouse modes and their correlation of runs and chains of unlike length, all staged in
    shared memory, as fast as two threads can ask for them."""
    import torch

    from paper_0903_5067_gb300 import analysis as an

    rng = np.random.default_rng(1)
    runs = [torch.tensor(rng.normal(size=s).cumsum(axis=1), device="cuda") for s in [(3000, 20, 3), (1700, 30, 3)]]
    chains = [torch.tensor(rng.normal(size=s).cumsum(axis=1), device="cuda") for s in [(4, 1100, 3), (4, 500, 3)]]
    want = [(torch.tensor(np.stack(an.msd(r, 2)), device="cuda"), an.rouse_modes(c, 2),
             torch.tensor(an.rouse_correlation(r, 200)[0], device="cuda")) for r, c in zip(runs, chains)]
    faults = []

    def work(q):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                s = torch.cuda.current_stream().cuda_stream
                out = [torch.empty_like(w) for w in want[q]]
                r, c, (g, X, m) = runs[q].data_ptr(), chains[q].data_ptr(), [o.data_ptr() for o in out]
                (T, N), M = runs[q].shape[:2], chains[q].shape[1]
                for _ in range(20):
                    for _ in range(100):
                        lblib.lb_analysis_rouse_modes(c, 4, M, 2, X, s)
                        lblib.lb_analysis_msd(r, T, N, 2, (N - 1) // 2, N // 2, g, s)
                    lblib.lb_analysis_rouse_correlation(r, T, N, 200, m, s)
                    torch.cuda.current_stream().synchronize()
                    assert all(torch.equal(a, b) for a, b in zip(out, want[q]))
        except Exception as e:
            faults.append(e)

    threads = [threading.Thread(target=work, args=(q,)) for q in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not faults, faults[0]
