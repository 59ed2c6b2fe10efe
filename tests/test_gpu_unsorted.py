"""Pushes of particles that are not in cell order: the deposit's other branch in 3D, and the steps
that do not count for a sort in 2D."""
import numpy as np
import pytest

from paper_1311_2286_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _order(w, kind, rng):
    """The workload's particles in cell order, in runs of two cells' length, or in random order, and
    with dead slots (cells outside the grid) among them."""
    for ps in w.particles:
        o = np.argsort(ps.cell, kind="stable")
        if kind == "random":
            rng.shuffle(o)
        elif kind == "pieces":  # long and short runs in one warp
            pieces = np.array_split(o, max(1, len(o) // 9))
            rng.shuffle(pieces := list(pieces))
            o = np.concatenate(pieces)
        ps.cell, ps.t, ps.v = ps.cell[o].copy(), ps.t[:, o].copy(), ps.v[:, o].copy()
        if kind != "sorted":
            ps.cell[::13] = w.n[0] + 1
    return w


def _records(run, s):
    cell, t, v = run.particles(s)
    return np.sort(np.rec.fromarrays([cell] + list(t) + list(v)))


@pytest.mark.parametrize("kind", ["sorted", "pieces", "random"])
@pytest.mark.parametrize("grid", [(8, 8, 8), (12, 20, 8), (16, 32), (72, 40)])
def test_any_order_gives_the_same_particles_and_charge(cpic, grid, kind):
    """Direct and tiled deposits, with and without a sort that counts in the push: whole numbers and
    particles are the same whatever order the particles come in."""
    got = []
    for tile, interval in ((0, 0), (1, 0), (0, 1), (1, 1)):
        rng = np.random.default_rng(17)
        mk = wl.sphere if len(grid) == 3 else wl.cylinder
        w = _order(mk(*grid, npart_per_species=20_001), kind, rng)
        run = cpic.run_from_workload(w, sort_interval=interval)
        run.set_push_tuning(0, tile)
        run.set_phi(wl.random_field(np.random.default_rng(4), tuple(reversed(run.n)), 0.5))
        run.step_particles(3)
        got.append([(_records(run, s), run.charge(s)) for s in range(2)])
        run.close()
    for other in got[1:]:
        for (a, qa), (b, qb) in zip(got[0], other):
            assert np.array_equal(a, b) and np.array_equal(qa, qb)
