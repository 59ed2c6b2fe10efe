"""The solver forms, the step's sort and the device hand-over at the sizes where they can go
wrong: tile and slab remainders, the smallest and the largest grid of a form, odd counts.

Tolerances: field solves 1e-10 relative L2 against the oracle's direct solve (solved to 1e-13, as
everywhere in this suite), or the oracle operator's residual where a direct solve is out of reach;
particles, counts and charges exact. A solve that ends above 1e-13 has reached the rounding of its
FP64 residual (cells seven times as long as wide): the error bound is the test."""
import ctypes
import math

import numpy as np
import pytest

from oracle import geometry, inject, poisson
from paper_1311_2286_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

P, Dr, Ne = 0, 1, 2
PP, PA, PR = 0, 1, 2
WALLS = [Dr, Dr, P, P]


def _solve(cpic, X, bc, bv, solver=None, axisym=False, npart=20_000):
    """Device solve to 1e-13 of a random charge; returns phi, the oracle's problem and the result."""
    D = X.shape[-1]
    n = tuple(X.shape[D - 1 - a] - 1 for a in range(D))
    g = geometry.build_geometry(X, [bc[2 * a] == P for a in range(D)], axisym=axisym)
    M, bbc = poisson.assemble(g, bc, bv)
    rng = np.random.default_rng(21)
    idx = np.stack([rng.integers(0, n[a], npart) for a in range(D)])
    t = rng.random((D, npart)).astype(np.float32)
    pbc = [PP if b == P else (PR if axisym or (D == 3 and b == Ne) else PA) for b in bc]
    cfg = cpic.make_config(D, n, bc, bv, pbc, 0.1, [(-1.0, 1.0, 1e-3, npart)], background=0.3, axisymmetric=axisym)
    run = cpic.Run(cfg)
    run.set_map_vertices(X)
    if solver is not None:
        run.set_solver(solver)
    run.load_particles(0, wl.pack_cells(idx), t, np.zeros((3, npart), np.float32))
    run.deposit()
    cycles, res = run.solve_field(rtol=1e-13, max_cycles=300, allow_not_converged=True)
    phi, C = run.phi(), run.charge(0)
    run.close()
    return phi, (g, M, bbc, poisson.charge_in_cells(g, [C], [-1e-3], 0.3)), (cycles, res)


SOLVES = {
    # cluster solver: slabs of four rows, slabs of six, a wide grid with short slabs, an Omega = r grid, a
    # singular one
    "slabs_of_4": (lambda: wl.annulus_vertices(32, 64, 1.0, 20.0), WALLS, [-5.0, 0, 0, 0], False, False),
    "slabs_of_6": (lambda: wl.annulus_vertices(64, 96, 1.0, 20.0), WALLS, [-5.0, 0, 0, 0], False, False),
    "wide": (lambda: wl.annulus_vertices(192, 64, 1.0, 40.0), WALLS, [-5.0, 0, 0, 0], False, False),
    "omega_r": (lambda: wl.sphere_axisym_vertices(32, 96, 1.0, 10.0), [Dr, Dr, Ne, Ne], [-2.5, 0, 0, 0], True, False),
    "singular": (lambda: wl.map2_vertices(64, 64, 0.0), [P] * 4, [0.0] * 4, False, False),
    # a grid of the cluster solver's outer iteration for which no slab layout fits
    "no_layout": (lambda: wl.annulus_vertices(192, 128, 1.0, 40.0), WALLS, [-5.0, 0, 0, 0], False, False),
    # launches per level: sizes that are no multiple of the 32 x 16 tile of the fused levels, and one
    # tile and a little
    "tile_remainders": (lambda: wl.annulus_vertices(72, 88, 1.0, 20.0), WALLS, [-5.0, 0, 0, 0], False, True),
    "narrow": (lambda: wl.map2_vertices(20, 136, 0.0), [Ne, Dr, P, P], [0, 1.0, 0, 0], False, True),
    "long_rows": (lambda: wl.annulus_vertices(136, 36, 1.0, 20.0), WALLS, [-5.0, 0, 0, 0], False, True),
    # the whole solve in one CTA: five and nine points, singular, small, and close to its 2048 cells
    "one_cta_5pt": (lambda: wl.annulus_vertices(34, 58, 1.0, 20.0), WALLS, [-5.0, 0, 0, 0], False, True),
    "one_cta_9pt": (lambda: wl.map2_vertices(20, 28, 0.08), [Dr, Ne, Dr, Dr], [0.3, 0, -1.0, 2.0], False, True),
    "one_cta_singular": (lambda: wl.map2_vertices(12, 44, 0.05), [P] * 4, [0.0] * 4, False, True),
    # and the first size above them
    "above_one_cta": (lambda: wl.map2_vertices(36, 60, 0.08), [P, P, Dr, Ne], [0, 0, 0.5, 0], False, True),
}


@pytest.mark.parametrize("case", list(SOLVES))
def test_solver_forms_at_their_edges(cpic, case, monkeypatch):
    mk, bc, bv, axisym, chain = SOLVES[case]
    monkeypatch.delenv("CPIC_NO_CLUSTER_SOLVER", raising=False)
    if chain:
        monkeypatch.setenv("CPIC_NO_CLUSTER_SOLVER", "1")
    for solver in (None, cpic.CPIC_SOLVER_MG) if chain else (None,):
        phi, (g, M, bbc, Q), (cycles, res) = _solve(cpic, mk(), bc, bv, solver, axisym)
        ref = poisson.solve(g, M, bbc, Q, bc)
        err = np.linalg.norm(phi - ref) / np.linalg.norm(ref)
        assert err <= 1e-10, (err, cycles, res)


@pytest.mark.parametrize("n", [(12, 12, 12), (8, 6, 10), (20, 12, 20), (40, 32, 40)])
def test_solver_forms_3d_at_their_edges(cpic, n):
    """The whole solve in one CTA, planes that do not divide evenly over the cluster's CTAs, and the
    per-level launches above the cluster part (rows that are no multiple of a block's)."""
    X = wl.shell_vertices(*n, 1.0, 30.0, math.pi / 32)
    bc, bv = [Dr, Dr, Ne, Ne, P, P], [-5.0, 0.0, 0.0, 0.0, 0.0, 0.0]
    for solver in (cpic.CPIC_SOLVER_BICGSTAB, cpic.CPIC_SOLVER_MG):
        phi, (g, M, bbc, Q), (cycles, res) = _solve(cpic, X, bc, bv, solver)
        if np.prod(n) > 20_000:
            r = poisson.residual_norm(M, bbc, g, Q, phi, bc)
            assert r <= 1e-10, (r, cycles, res)
            continue
        ref = poisson.solve(g, M, bbc, Q, bc)
        err = np.linalg.norm(phi - ref) / np.linalg.norm(ref)
        assert err <= 1e-10, (err, cycles, res)


def _records(run, s):
    cell, t, v = run.particles(s)
    return cell, np.sort(np.rec.fromarrays([cell] + list(t) + list(v)))


SORTS = {
    "one_particle": (lambda: wl.cylinder(16, 32, npart_per_species=1, inject=False, capacity_factor=4.0), {}),
    "chunk_and_one": (lambda: wl.cylinder(64, 128, npart_per_species=8193, inject=True, capacity_factor=2.0), {}),
    "odd": (lambda: wl.cylinder(72, 128, npart_per_species=70_001, inject=True), {"chunk": 768}),
    "direct": (lambda: wl.cylinder(24, 40, npart_per_species=30_003, inject=True), {"tile": 0}),
    "sphere_direct": (lambda: wl.sphere(16, 12, 20, npart_per_species=20_001, inject=True), {"tile": 0}),
    "sphere_empty_species": (lambda: wl.sphere(8, 8, 8, npart_per_species=3, capacity_factor=40.0), {"tile": 0}),
}


@pytest.mark.parametrize("case", list(SORTS))
def test_sorted_steps_keep_the_particles(cpic, case):
    """A step's push and injection number the particles of each cell, and the sort is a look-up of
    the slots: three steps sorted each time hold the same particles and charge as three without a
    sort, in cell order, also where a read comes between the sort and the push that carries it out."""
    mk, tune = SORTS[case]
    runs = []
    for interval in (0, 1):
        run = cpic.run_from_workload(mk(), sort_interval=interval)
        run.set_push_tuning(tune.get("chunk", 0), tune.get("tile", 1))
        run.set_phi(wl.random_field(np.random.default_rng(4), tuple(reversed(run.n)), 0.5))
        run.step_particles(2)
        if interval:
            run.particles(0)
        run.step_particles(1)
        runs.append(run)
    plain, sorted_ = runs
    a, b = plain.diag(), sorted_.diag()
    for s in range(2):
        _, ra = _records(plain, s)
        cell, rb = _records(sorted_, s)
        assert np.array_equal(ra, rb)
        assert np.array_equal(plain.charge(s), sorted_.charge(s))
        assert a["absorbed"][s] == b["absorbed"][s] and a["injected"][s] == b["injected"][s]
        idx = wl.unpack_cells(cell, len(plain.n))
        key = idx[0].astype(np.int64)
        stride = 1
        for ax in range(1, len(plain.n)):
            stride *= plain.n[ax - 1]
            key = key + stride * idx[ax].astype(np.int64)
        assert np.all(np.diff(key) >= 0)
    for run in runs:
        run.close()


@pytest.mark.parametrize("D,n", [(2, 1), (2, 31), (2, 4097), (3, 255), (3, 1026)])
def test_device_arrays_equal_host_arrays(cpic, D, n):
    """Loads from and reads into device arrays give what the host arrays give, invalid particles
    (dropped) and dead slots included."""
    torch = pytest.importorskip("torch")
    w = wl.cylinder(16, 32, npart_per_species=n) if D == 2 else wl.sphere(8, 8, 8, npart_per_species=n)
    cfg = cpic.config_from_workload(w)
    cell, t, v = (np.ascontiguousarray(x) for x in (w.particles[0].cell, w.particles[0].t, w.particles[0].v))
    cell = cell.copy()
    if n > 30:
        cell[n // 2] = (w.n[0] + 3) | (1 << (16 if D == 2 else 10))  # outside the grid
    out = []
    for device in (False, True):
        run = cpic.Run(cfg)
        run.set_map_vertices(w.vertices)
        if device:
            run.load_particles(0, *(torch.from_numpy(x).cuda() for x in (cell, t, v)))
        else:
            run.load_particles(0, cell, t, v)
        run.set_phi(wl.random_field(np.random.default_rng(5), tuple(reversed(w.n)), 0.5))
        run.vertex_field()
        run.push()
        cap = int(cfg.capacity[0])
        m = ctypes.c_int64()
        if device:
            bufs = [torch.empty(k * cap, dtype=d, device="cuda") for k, d in
                    ((1, torch.int32), (D, torch.float32), (3, torch.float32))]
            cpic.check(cpic.load().cpic_get_particles(run.h, 0, cap, ctypes.byref(m),
                                                      *(ctypes.c_void_p(b.data_ptr()) for b in bufs)))
            run.synchronize()
            k = m.value
            out.append([b.cpu().numpy()[: c * k].reshape(c, k) for b, c in zip(bufs, (1, D, 3))])
        else:
            c, tt, vv = run.particles(0)
            out.append([c.reshape(1, -1), tt, vv])
        run.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("drift", [-6.0, -0.05, 0.05, 2.5])
def test_drifting_inversion_over_the_drifts(cpic, drift):
    """The normal speed of a drifting inflow, for drifts from deep inflow to well out of the domain
    (drift in thermal speeds along x; the face is xi = 1, whose inward normal is -x)."""
    w = wl.planar_wall(16, 8, ppc=4000)
    g = geometry.build_geometry(w.vertices, [False, True])
    vth, seed = 1.0, 91
    d3 = (drift * vth, 0.2, 0.0)
    wts = inject.face_drift_weights_2d(w.vertices, g.k, 1, d3, vth)
    tot = 0.0
    for x in wts:
        tot += float(x)
    sp = w.species[0]
    dens = 1500.5 * sp.w / (tot * w.dt)
    w.injection = [(0, 1, dens, vth, seed, d3)]
    run = cpic.run_from_workload(w)
    run.vertex_field()
    run.push()
    run.inject()
    c, t, v = run.particles(0)
    run.close()
    cnt = inject.count_at_step(dens * tot * w.dt / sp.w, 0)
    assert cnt == 1500
    idx, t32, v32, keep = inject.inject_2d(g.k, w.n, 1, cnt, 0, 0, seed, vth, d3, w.dt, drift_weights=wts)
    assert c.shape[0] == int(keep.sum())
    ok = c == wl.pack_cells(idx)
    assert np.sum(~ok) <= 1
    np.testing.assert_allclose(v[:, ok], v32[:, ok], rtol=2e-6, atol=2e-6 * vth)
    np.testing.assert_allclose(t[:, ok], t32[:, ok], atol=1e-5)


@pytest.mark.parametrize("shifted", [0, 1, 2])
def test_device_arrays_off_their_words_are_copied(cpic, shifted):
    """A device array at an odd byte address (cell, t or v) loads and reads as it does at a word."""
    torch = pytest.importorskip("torch")
    n = 1000
    w = wl.cylinder(16, 32, npart_per_species=n)
    arrays = [np.ascontiguousarray(x) for x in (w.particles[0].cell, w.particles[0].t, w.particles[0].v)]
    run = cpic.Run(cpic.config_from_workload(w))
    run.set_map_vertices(w.vertices)

    def room(k, nbytes):
        at = 2 if k == shifted else 0
        return torch.zeros(nbytes + 64, dtype=torch.uint8, device="cuda")[at:at + nbytes]

    bufs = [room(k, x.nbytes) for k, x in enumerate(arrays)]
    for b, x in zip(bufs, arrays):
        b.copy_(torch.from_numpy(x.reshape(-1).view(np.uint8)))
    torch.cuda.synchronize()
    ptrs = [ctypes.c_void_p(b.data_ptr()) for b in bufs]
    assert ptrs[shifted].value % 4 == 2
    cpic.check(cpic.load().cpic_load_particles(run.h, 0, n, *ptrs))
    run.synchronize()
    for a, b in zip(run.particles(0), arrays):
        assert np.array_equal(a.reshape(-1), b.reshape(-1))
    for b in bufs:
        b.zero_()
    torch.cuda.synchronize()
    m = ctypes.c_int64()
    cpic.check(cpic.load().cpic_get_particles(run.h, 0, n, ctypes.byref(m), *ptrs))
    run.synchronize()
    assert m.value == n
    for b, x in zip(bufs, arrays):
        assert np.array_equal(b.cpu().numpy(), x.reshape(-1).view(np.uint8))
    run.close()
