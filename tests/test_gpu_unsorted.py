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


@pytest.mark.parametrize("grid", [(12, 20, 8), (72, 40)])
def test_a_run_without_room_for_the_numbers_sorts_all_the_same(cpic, grid):
    """An arena that has no room for the particles' numbers is taken, and a run made without a sort
    interval may be given one: the particles and their order by cell are those of a run with numbers."""
    torch = pytest.importorskip("torch")
    mk = wl.sphere if len(grid) == 3 else wl.cylinder
    got = []
    for how in ("numbers", "small_arena", "interval_later"):
        w = mk(*grid, npart_per_species=20_001, inject=True)
        small = cpic.Run.footprint(cpic.config_from_workload(w, sort_interval=0))
        arena = torch.empty(small, dtype=torch.uint8, device="cuda") if how != "numbers" else None
        run = cpic.run_from_workload(w, sort_interval=0 if how == "interval_later" else 1, arena=arena)
        if how == "interval_later":
            run.set_sort_interval(1)
        run.set_push_tuning(0, 0)
        run.set_phi(wl.random_field(np.random.default_rng(4), tuple(reversed(run.n)), 0.5))
        run.step_particles(3)
        got.append([(run.particles(s)[0], _records(run, s), run.charge(s)) for s in range(2)])
        run.close()
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert all(np.array_equal(x, y) for x, y in zip(a, b))
    with pytest.raises(cpic.CpicError) as e:
        cpic.Run(cpic.config_from_workload(w, sort_interval=1), arena=torch.empty(small - 256, dtype=torch.uint8,
                                                                                 device="cuda"))
    assert e.value.status == -2
