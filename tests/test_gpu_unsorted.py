"""Pushes of particles that are not in cell order: the deposit's other branch in 3D, and the steps
that do not count for a sort in 2D."""
import ctypes

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
def test_a_run_without_room_for_the_numbers_sorts_all_the_same(cpic, grid, tmp_path):
    """A run made without a sort interval may be given one, and restored into its arena from then: the
    particles and their order by cell are those of a run with room for the numbers. (A new run with
    an interval needs that room.)"""
    torch = pytest.importorskip("torch")
    mk = wl.sphere if len(grid) == 3 else wl.cylinder
    got = []
    for how in ("numbers", "interval_later", "restored"):
        w = mk(*grid, npart_per_species=20_001, inject=True)
        small = cpic.Run.footprint(cpic.config_from_workload(w, sort_interval=0))
        arena = torch.empty(small, dtype=torch.uint8, device="cuda") if how != "numbers" else None
        run = cpic.run_from_workload(w, sort_interval=1 if how == "numbers" else 0, arena=arena)
        if how != "numbers":
            run.set_sort_interval(1)
        run.set_push_tuning(0, 0)
        run.set_phi(wl.random_field(np.random.default_rng(4), tuple(reversed(run.n)), 0.5))
        run.step_particles(2)
        if how == "restored":
            run.checkpoint(str(tmp_path / "state"))
            run.close()
            run.h = ctypes.c_void_p()
            cpic.check(cpic.load().cpic_restore(str(tmp_path / "state").encode(), ctypes.c_void_p(arena.data_ptr()),
                                                small, None, ctypes.byref(run.h)))
            run.set_push_tuning(0, 0)
        run.step_particles(1)
        got.append([(run.particles(s)[0], _records(run, s), run.charge(s)) for s in range(2)])
        run.close()
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert all(np.array_equal(x, y) for x, y in zip(a, b))
    with pytest.raises(cpic.CpicError) as e:
        cpic.Run(cpic.config_from_workload(w, sort_interval=1), arena=arena)
    assert e.value.status == -2
