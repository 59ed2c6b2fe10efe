"""What a field solve reports when it cannot end well, or has nothing to do, in each of its forms."""
import math

import numpy as np
import pytest

from paper_1311_2286_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

P, Dr, Ne = 0, 1, 2
PP, PA, PR = 0, 1, 2
WALLS = [Dr, Dr, P, P]
SHELL = [Dr, Dr, Ne, Ne, P, P]
NOT_CONVERGED = -4

# vertices, field boundaries, off the cluster solver, outer iteration (None: the default)
FORMS = {
    "cluster": (lambda: wl.annulus_vertices(64, 96, 1.0, 20.0), WALLS, False, None),
    "v_cycles_without_a_layout": (lambda: wl.annulus_vertices(192, 128, 1.0, 40.0), WALLS, False, None),
    "launches": (lambda: wl.annulus_vertices(72, 88, 1.0, 20.0), WALLS, True, None),
    "launches_v_cycles": (lambda: wl.annulus_vertices(72, 88, 1.0, 20.0), WALLS, True, "mg"),
    "one_cta": (lambda: wl.annulus_vertices(34, 58, 1.0, 20.0), WALLS, True, None),
    "one_cta_3d": (lambda: wl.shell_vertices(8, 6, 10, 1.0, 30.0, math.pi / 32), SHELL, False, None),
    "launches_3d": (lambda: wl.shell_vertices(20, 12, 20, 1.0, 30.0, math.pi / 32), SHELL, False, None),
    "launches_3d_v_cycles": (lambda: wl.shell_vertices(20, 12, 20, 1.0, 30.0, math.pi / 32), SHELL, False, "mg"),
}


@pytest.fixture(params=list(FORMS))
def form(request, cpic, monkeypatch):
    """A run of the form: (run, potential at the cells), with the given boundary value at xi = 0."""
    mk, bc, chain, solver = FORMS[request.param]
    monkeypatch.delenv("CPIC_NO_CLUSTER_SOLVER", raising=False)
    if chain:
        monkeypatch.setenv("CPIC_NO_CLUSTER_SOLVER", "1")
    runs = []

    def make(value):
        X = mk()
        D = X.shape[-1]
        n = tuple(X.shape[D - 1 - a] - 1 for a in range(D))
        pbc = [PP if b == P else (PR if b == Ne else PA) for b in bc]
        run = cpic.Run(cpic.make_config(D, n, bc, [value] + [0.0] * 5, pbc, 0.1, [(-1.0, 1.0, 1e-3, 64)],
                                        mg_max_cycles=6, mg_rtol=1e-10))
        run.set_map_vertices(X)
        if solver:
            run.set_solver(cpic.CPIC_SOLVER_MG)
        runs.append(run)
        return run, wl.random_field(np.random.default_rng(3), tuple(reversed(n)), 1.0)

    yield make
    for run in runs:
        run.close()


def _solve(cpic, run):
    try:
        return (0, *run.solve_field(rtol=1e-10, max_cycles=6))
    except cpic.CpicError as e:
        return e.status, None, None


@pytest.mark.parametrize("bad", [math.nan, math.inf])
def test_a_potential_that_is_no_number_does_not_converge(cpic, form, bad):
    run, phi = form(-5.0)
    phi.reshape(-1)[phi.size // 3] = bad
    run.set_phi(phi)
    assert _solve(cpic, run)[0] == NOT_CONVERGED
    run.set_phi(phi)
    run.step(1)
    d = run.diag()
    assert not d["mg_residual"] <= 1e-10 and d["mg_cycles"] == 6
    run.set_phi(np.zeros_like(phi))  # and the next solve starts afresh
    run.solve_field(rtol=1e-6, max_cycles=100)


@pytest.mark.parametrize("bad", [math.nan, math.inf])
def test_a_boundary_value_that_is_no_number_does_not_converge(cpic, form, bad):
    run, phi = form(bad)
    assert _solve(cpic, run)[0] == NOT_CONVERGED


def test_nothing_to_solve_ends_at_once(cpic, form):
    """A zero right-hand side (no particles, grounded walls) is within any tolerance: no cycle, the
    potential stays, in a solve and in a step."""
    run, phi = form(0.0)
    run.set_phi(phi)
    assert _solve(cpic, run) == (0, 0, 0.0)
    assert np.array_equal(run.phi(), phi)
    run.step(1)
    d = run.diag()
    assert d["mg_cycles"] == 0 and d["mg_residual"] == 0.0
    assert np.array_equal(run.phi(), phi)


# (the cluster kernel ends its own loop, and takes the residual of its last permitted cycle in FP64)
@pytest.mark.parametrize("form", [f for f in FORMS if f != "cluster"], indirect=True)
def test_a_cycle_enqueued_beyond_the_last_leaves_the_potential(cpic, form):
    """The cycle that a host one ahead has enqueued when the solve ends changes nothing: the potential
    is that of a solve cut off at the same number of cycles, and solving again does none."""
    run, phi = form(-5.0)
    run.set_phi(phi)
    cycles, res = run.solve_field(rtol=1e-9, max_cycles=100)
    first = run.phi()
    run.set_phi(phi)
    assert run.solve_field(rtol=1e-9, max_cycles=cycles) == (cycles, res)
    assert np.array_equal(run.phi(), first)
    assert run.solve_field(rtol=1e-9, max_cycles=100) == (0, res)
    assert np.array_equal(run.phi(), first)
