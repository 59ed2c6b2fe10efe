"""Performance cases: the calls a program makes of this library, over the sizes it is used at.

A case is a plasma (``kind``: a map with its species, boundaries and injection), a grid, a
number of macro-particles per species and what the program does with it (``do``):

  cycle     one whole PIC step (cpic_step): vertex field, push, deposit, injection, sort when
            it is due, field solve to the default tolerance; the new potential, the deposited
            charge and the diagnostics are read, then the prescribed potential is put back
            (test particles in a given field, with the potential of their charge monitored),
            so that every pass pushes in the same field;
  particles ``steps`` particle steps in a fixed field (cpic_step_particles), the charge and the
            diagnostics read at the end;
  handover  a caller that owns its particles: hands them over, takes one particle step, gets
            all of them back (storage order, no sort);
  batch     one step of a batch of uneven runs, whole cycles.

Particles are loaded on the device except where a test problem has a closed-form density
(map2), and start half a step back in the field (cpic_kick), as cpic_initialize does.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1311_2286_gb300 import cpic
from paper_1311_2286_gb300 import workloads as wl


def listed():
    return [
        # the Langmuir-wave test problem at its smallest: a launch-bound whole step with the
        # 9-point singular periodic solve
        dict(name="langmuir_32x32", kind="map2", do="cycle", n1=32, n2=32, n3=1, pps=65536, sort=4, steps=1),
        # the paper's mover timing (Tables II-III): 64 x 64 cells, 100 per cell, fixed field
        dict(name="map2_mover_64x64", kind="map2", do="particles", n1=64, n2=64, n3=1, pps=409600, sort=4, steps=10),
        # a coupled code that owns a million particles and passes them in and out each step
        dict(name="map2_handover_128x128", kind="map2", do="handover", n1=128, n2=128, n3=1, pps=1048576, sort=0,
             steps=1),
        # the planar wall (Test A): drifting ions injected, 64 per cell and species
        dict(name="wall_128x128", kind="wall", do="cycle", n1=128, n2=128, n3=1, pps=1048576, sort=4, steps=1),
        # the 2D cylinder in plasma, the usual size of a 2D production run
        dict(name="cylinder_128x256", kind="cylinder", do="cycle", n1=128, n2=256, n3=1, pps=2000000, sort=4, steps=1),
        # the large 2D cylinder: particles alone, and whole steps (a grid the one-cluster solver
        # does not take)
        dict(name="cylinder_512x1024_particles", kind="cylinder", do="particles", n1=512, n2=1024, n3=1, pps=32000000,
             sort=2, steps=2),
        dict(name="cylinder_512x1024", kind="cylinder", do="cycle", n1=512, n2=1024, n3=1, pps=8000000, sort=2,
             steps=1),
        # the magnetised sphere in (r, z) geometry (Test C): rings, exact gyration
        dict(name="axisym_128x128_B19", kind="axisym", do="cycle", n1=128, n2=128, n3=1, pps=3768320, sort=8, steps=1),
        # a small 3D run with the library's default push settings
        dict(name="sphere_24x20x16", kind="sphere", do="cycle", n1=24, n2=20, n3=16, pps=60013, sort=4, steps=1),
        # the headline: 3D sphere, 64M particles, the settings the autotuner picks there
        dict(name="sphere_128_particles", kind="sphere", do="particles", n1=128, n2=128, n3=128, pps=32000000, sort=1,
             steps=2, tuned=True),
        # whole steps on the same grid with a quarter of the particles
        dict(name="sphere_128", kind="sphere", do="cycle", n1=128, n2=128, n3=128, pps=8000000, sort=1, steps=1,
             tuned=True),
        # a parameter scan: eight uneven cylinders stepped together
        dict(name="batch_8", kind="cylinder", do="batch", n1=256, n2=512, n3=1, pps=2000000, sort=4, steps=1, runs=8,
             mix=1000),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges: grids coarse 2^p (coarse counts 4..9, odd ones among
    them), 4 to about 500 particles per cell and species up to the listed totals."""
    kind = rng.choice(["langmuir", "mover", "handover", "wall", "cylinder", "cylinder", "axisym", "sphere", "sphere",
                       "batch"])
    odd = rng.randrange(0, 2)
    if kind == "batch":
        return dict(kind="cylinder", do="batch", n1=256, n2=512, n3=1, pps=2000000, sort=rng.choice([2, 4, 8]), steps=1,
                    runs=rng.randrange(3, 9), mix=rng.randrange(1, 1 << 20))
    if kind == "sphere":
        p = rng.randrange(1, 5)
        n = [rng.randrange(4, 8) << p for _ in range(3)]
        cells = n[0] * n[1] * n[2]
        pps = int(min(_log(rng, 4.0, 64.0) * cells, 32e6)) | odd
        do = rng.choice(["cycle", "particles"])
        if do == "cycle":
            pps = min(pps, 8000000 + odd)
        return dict(kind="sphere", do=do, n1=n[0], n2=n[1], n3=n[2], pps=pps, sort=rng.choice([1, 2, 4]),
                    steps=1 if do == "cycle" else 2, tuned=rng.random() < 0.7)
    top = {"langmuir": 3, "mover": 5, "handover": 5, "wall": 5, "cylinder": 6, "axisym": 5}[kind]
    p = rng.randrange(2, top + 1)
    n1, n2 = rng.randrange(4, 10) << p, rng.randrange(4, 17 if kind == "cylinder" else 10) << p
    cells = n1 * n2
    pps = int(min(_log(rng, 16.0, 512.0) * cells, 2.0e7)) | odd
    if kind in ("langmuir", "mover", "handover"):
        pps = min(pps, 2000000 + odd)
        do = {"langmuir": "cycle", "mover": "particles", "handover": "handover"}[kind]
        return dict(kind="map2", do=do, n1=n1, n2=n2, n3=1, pps=pps, sort=0 if do == "handover" else 4,
                    steps=10 if do == "particles" else 1)
    do = rng.choice(["cycle", "particles"]) if kind == "cylinder" else "cycle"
    return dict(kind=kind, do=do, n1=n1, n2=n2, n3=1, pps=min(pps, 8000000 + odd) if do == "cycle" else pps,
                sort=rng.choice([2, 4, 8]), steps=1 if do == "cycle" else 2)


# ------------------------------------------------------------------ what a program sets up


def _workload(case, seed):
    """The case's plasma with the potential it is pushed in: the vacuum or
    linear solution of its problem, at the cell centres."""
    n1, n2, n3, pps = case["n1"], case["n2"], case["n3"], case["pps"]
    xi = (np.arange(n1) + 0.5) / n1
    if case["kind"] == "map2":
        w = wl.langmuir_map2(n1, n2, ppc=1, vth=0.05, seed=seed)
        w.species[0].w, w.species[0].capacity = 1.0 / pps, pps
        w.particles = [wl.load_map2(np.random.default_rng(seed), n1, n2, 0.05, pps, 0.05, amp=0.01)]
        xc = w.vertices[..., 0]
        xc = 0.25 * (xc[:-1, :-1] + xc[1:, :-1] + xc[:-1, 1:] + xc[1:, 1:])
        phi = -0.01 / (2.0 * math.pi) ** 2 * np.cos(2.0 * math.pi * xc)
    elif case["kind"] == "wall":
        w = wl.planar_wall(n1, n2, ppc=pps / (n1 * n2), seed=seed % 100000)
        w.field_bc_value[0] = -2.1  # the wall at its steady state
        phi = np.broadcast_to(-2.1 * np.exp(-20.0 * xi), (n2, n1))
    elif case["kind"] == "cylinder":
        w = wl.cylinder(n1, n2, npart_per_species=pps, seed=seed % 100000, host_particles=False)
        phi = np.broadcast_to(-5.0 * (1.0 - xi), (n2, n1))
    elif case["kind"] == "axisym":
        w = wl.sphere_axisym(n1, n2, npart_per_species=8, seed=seed % 100000, dt=0.05)
        for s in w.species:
            s.w, s.capacity = s.w * 8.0 / pps, int(1.5 * pps)
        w.particles = [wl.ParticleSet(p.cell[:0], p.t[:, :0], p.v[:, :0]) for p in w.particles]
        w.B0, w.gyro = (0.0, 19.0, 0.0), "cyclotronic"
        r = 1.0 + 9.0 * xi
        phi = np.broadcast_to(-2.5 * (1.0 / r - 0.1) / 0.9, (n2, n1))
    else:
        w = wl.sphere(n1, n2, n3, npart_per_species=pps, seed=seed % 100000, host_particles=False, inject=True)
        r = 30.0 ** xi
        phi = np.broadcast_to(-5.0 * (1.0 / r - 1.0 / 30.0) / (1.0 - 1.0 / 30.0), (n3, n2, n1))
    return w, np.ascontiguousarray(phi)


_ANALYTIC = {"cylinder": (cpic.CPIC_MAP_ANNULUS, [1.0, 40.0]), "sphere": (cpic.CPIC_MAP_SHELL, [1.0, 30.0, math.pi / 32]),
             "axisym": (cpic.CPIC_MAP_SPHERE_AXISYM, [1.0, 10.0]), "map2": (cpic.CPIC_MAP_SINE, [0.05])}


def _at(tensor):
    return ctypes.c_void_p(tensor.data_ptr())


class _State:
    batch = None

    def __del__(self):
        if self.batch is not None:  # before its member runs
            self.batch.close()


def _start(run, w, phi, seed, host):
    """Particles in cell order, half a step back in the field phi."""
    for s, sp in enumerate(w.species):
        if host:
            ps = w.particles[s]
            run.load_particles(s, ps.cell, ps.t, ps.v)
        else:
            drift = [w.injection[s][5][0], 0.0, 0.0] if w.injection and len(w.injection[s]) > 5 else None
            run.load_maxwellian(s, w.pps, sp.vth, seed=seed * 16 + s, drift=drift)
    run.set_phi(phi)
    run.vertex_field()
    run.kick(-0.5)


def prepare(case, seed):
    st = _State()
    st.case = case
    if case["do"] == "batch":
        st.runs, st.phi = [], []
        st.batch = cpic.Batch(case["runs"])
        for i, spec in enumerate(wl.batch_specs(case["runs"], seed=case["mix"])):
            spec["seed"] = seed % 100000 + i
            run = cpic.cylinder_run_device(**spec, sort_interval=case["sort"])
            w, phi = _workload(dict(case, n1=spec["n1"], n2=spec["n2"], pps=spec["npart_per_species"]), spec["seed"])
            w.pps = spec["npart_per_species"]
            phi = phi * (spec["phi_obj"] / -5.0)
            _start(run, w, phi, spec["seed"], False)
            run.sort()
            st.batch.add(run)
            st.runs.append(run)
            st.phi.append(torch.from_numpy(phi).cuda())
        return st
    w, phi = _workload(case, seed)
    w.pps = case["pps"]
    host = case["kind"] == "map2"
    cfg = cpic.config_from_workload(w, sort_interval=case["sort"])
    st.arena = torch.empty(cpic.Run.footprint(cfg), dtype=torch.uint8, device="cuda")
    run = st.run = cpic.Run(cfg, arena=st.arena)
    if case["kind"] in _ANALYTIC:
        run.set_map_analytic(*_ANALYTIC[case["kind"]])
    else:
        run.set_map_vertices(w.vertices)
    if w.B0 is not None:
        run.set_magnetic_field(w.B0)
        run.set_gyro_integrator(w.gyro)
    if case.get("tuned"):  # what cpic_autotune picks on the large spheres
        run.set_push_tuning(8192 if case["pps"] > 4000000 else 0, 0)
    if case["do"] == "handover":
        ps = w.particles[0]
        order = np.argsort(ps.cell, kind="stable")
        st.particles = [torch.from_numpy(np.ascontiguousarray(a)).cuda()
                        for a in (ps.cell[order], ps.t[:, order], ps.v[:, order])]
        run.set_phi(phi)
        return st
    _start(run, w, phi, seed % 100000, host)
    run.sort()
    for inj in w.injection:
        run.set_injection(*inj[:5], drift=inj[5] if len(inj) > 5 else None)
    st.phi = torch.from_numpy(phi).cuda()
    return st


def _read(run, solved):
    """What a program reads after its steps: the charge of every species, the potential when it
    was solved for, energies and particle counts."""
    lib, out = cpic.load(), {}
    if solved:
        out["phi"] = torch.empty(run.ncell, dtype=torch.float64, device="cuda")
        cpic.check(lib.cpic_get_phi(run.h, _at(out["phi"])))
    for s in range(run.cfg.n_species):
        q = out["charge%d" % s] = torch.empty(run.ncell, dtype=torch.int64, device="cuda")
        cpic.check(lib.cpic_get_charge(run.h, s, _at(q)))
    d = run.diag()
    out["counts"] = [d["n"], d["absorbed"], d["injected"], d["dropped"], d["nonfinite"]]
    out["kinetic"] = d["W_K"]
    if solved:
        out["field"] = d["W_E"]
    return out


def run(st):
    case = st.case
    lib = cpic.load()
    if case["do"] == "batch":
        st.batch.step(case["steps"], solve=True)
        st.batch.synchronize()
        out = []
        for r, phi in zip(st.runs, st.phi):
            got = _read(r, True)
            out.append([got["phi"], got["charge0"], got["charge1"]])
            cpic.check(lib.cpic_set_phi(r.h, _at(phi)))
        return out
    r = st.run
    if case["do"] == "handover":
        r.load_particles(0, *st.particles)
        r.step_particles(1)
        out = [torch.empty_like(a) for a in st.particles]
        n = ctypes.c_int64()
        cpic.check(lib.cpic_get_particles(r.h, 0, out[0].shape[0], ctypes.byref(n), *map(_at, out)))
        return out
    if case["do"] == "particles":
        r.step_particles(case["steps"])
        return _read(r, False)
    r.step(case["steps"])
    out = _read(r, True)
    cpic.check(lib.cpic_set_phi(r.h, _at(st.phi)))
    return out


def work(case):
    """Every particle's state read and written once per step, the potential read and each
    species' charge written once; a cycle also reads the charge and writes the potential. The
    arithmetic is the mover's and the deposit's (two gathers, predictor and corrector, node
    weights); the solve's depends on the method and is left out."""
    if case["do"] == "batch":
        specs = wl.batch_specs(case["runs"], seed=case["mix"])
        runs = [(s["n1"] * s["n2"], 2 * s["npart_per_species"]) for s in specs]
    else:
        nsp = 1 if case["kind"] == "map2" else 2
        runs = [(case["n1"] * case["n2"] * case["n3"], nsp * case["pps"])]
    D = 3 if case["kind"] == "sphere" else 2
    solved = case["do"] in ("cycle", "batch")
    nsp = 1 if case["kind"] == "map2" else 2
    cells, parts = sum(c for c, _ in runs), sum(p for _, p in runs)
    grid = 8 * cells * (1 + nsp) + (8 * cells * (1 + nsp) if solved else 0)
    return {"bytes": case["steps"] * (2 * (16 + 4 * D) * parts + grid),
            "flops": case["steps"] * parts * (150 if D == 2 else 500)}


# ------------------------------------------------------------------ 64-bit values (map2)


def _metric(n1, n2, eps, dev):
    """k = du/dx at the vertices (cell units), cell areas, face coefficients J g^{ab} of the
    periodic map2 square, by finite differences of the vertex map, arrays [j, i]."""
    v = torch.from_numpy(wl.map2_vertices(n1, n2, eps)).to(dev)
    x = v[:-1, :-1]
    px = torch.tensor([1.0, 0.0], dtype=torch.float64, device=dev)
    py = torch.tensor([0.0, 1.0], dtype=torch.float64, device=dev)

    def diff(a, axis, period):  # a[+1] - a[0] with the period at the seam
        d = torch.roll(a, -1, axis) - a
        idx = [slice(None)] * 3
        idx[axis] = -1
        d[tuple(idx)] += period
        return d

    ex, ey = diff(x, 1, px), diff(x, 0, py)  # edges from vertex (j, i)
    du, dv = 0.5 * (ex + torch.roll(ex, 1, 1)), 0.5 * (ey + torch.roll(ey, 1, 0))
    cross = lambda a, b: a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0]  # noqa: E731
    det = cross(du, dv)
    k = torch.stack([dv[..., 1], -dv[..., 0], -du[..., 1], du[..., 0]], -1) / det[..., None]
    area = cross(0.5 * (ex + torch.roll(ex, -1, 0)), 0.5 * (ey + torch.roll(ey, -1, 1)))
    fu = 0.5 * (du + torch.roll(du, -1, 0))  # faces normal to xi: vertex (j, i) to (j+1, i)
    fv = 0.5 * (dv + torch.roll(dv, -1, 1))
    ju, jv = cross(fu, ey), cross(ex, fv)
    a = {"uu": (ey * ey).sum(-1) / ju, "uv": -(fu * ey).sum(-1) / ju,
         "vv": (ex * ex).sum(-1) / jv, "vu": -(ex * fv).sum(-1) / jv}
    return k, area, a


def _step64(n, k, phi, cell, t, v, dt, qm):
    """One step of the hybrid mover in 64 bits (periodic); cells as floats, arrays [2, N]."""
    n2, n1 = phi.shape
    west, south = torch.roll(phi, 1, 1), torch.roll(phi, 1, 0)
    both = torch.roll(west, 1, 0)
    g = torch.stack([0.5 * ((south - both) + (phi - west)), 0.5 * ((west - both) + (phi - south))], -1)

    def gather(tab, c, f):
        i, j = c[0].long() % n1, c[1].long() % n2
        i1, j1 = (i + 1) % n1, (j + 1) % n2
        w = [(1 - f[0]) * (1 - f[1]), f[0] * (1 - f[1]), (1 - f[0]) * f[1], f[0] * f[1]]
        return sum(a[:, None] * tab[b] for a, b in zip(w, [(j, i), (j, i1), (j1, i), (j1, i1)])).T

    kp, gp = gather(k, cell, t), gather(g, cell, t)
    new = v.clone()
    new[0] -= dt * qm * (gp[0] * kp[0] + gp[1] * kp[2])
    new[1] -= dt * qm * (gp[0] * kp[1] + gp[1] * kp[3])
    move = lambda kk: torch.stack([kk[0] * new[0] + kk[1] * new[1], kk[2] * new[0] + kk[3] * new[1]])  # noqa: E731
    x = t + 0.5 * dt * move(kp)
    kq = gather(k, cell + torch.floor(x), x - torch.floor(x))
    x = t + dt * move(kq)
    size = torch.tensor([[float(n1)], [float(n2)]], dtype=torch.float64, device=phi.device)
    return torch.remainder(cell + torch.floor(x), size), x - torch.floor(x), new, (v * new).sum()


def _solve64(n1, n2, area, a, cell, t, w):
    """The potential of electrons of weight w in a neutralising background: quadratic-spline
    charge, conservative finite volumes, dense solve, gauge sum J phi = 0; and its energy."""
    i, j = cell[0].long(), cell[1].long()
    count = torch.zeros(n2, n1, dtype=torch.float64, device=t.device)
    s = [[0.5 * (1 - f) ** 2, 0.75 - (f - 0.5) ** 2, 0.5 * f**2] for f in t]
    for q in range(3):
        for p in range(3):
            count.index_put_(((j + q - 1) % n2, (i + p - 1) % n1), s[0][p] * s[1][q], accumulate=True)
    charge = area - w * count
    e = torch.eye(n1 * n2, dtype=torch.float64, device=t.device).reshape(n2, n1, n1 * n2)
    west, south = torch.roll(e, 1, 1), torch.roll(e, 1, 0)
    su, sv = e + west, e + south
    flux = a["uu"][..., None] * (e - west) + 0.25 * a["uv"][..., None] * (torch.roll(su, -1, 0) - torch.roll(su, 1, 0))
    flvx = a["vv"][..., None] * (e - south) + 0.25 * a["vu"][..., None] * (torch.roll(sv, -1, 1) - torch.roll(sv, 1, 1))
    m = -((torch.roll(flux, -1, 1) - flux) + (torch.roll(flvx, -1, 0) - flvx)).reshape(n1 * n2, n1 * n2)
    J = area.reshape(-1)
    b = charge.reshape(-1) - charge.sum() / J.sum() * J
    phi = torch.linalg.solve(m + J[None, :], b)  # adds (sum J phi), zero in the gauge
    phi = phi - (J * phi).sum() / J.sum()
    return phi, 0.5 * float((phi * charge.reshape(-1)).sum())


def exact(case, seed):
    """64-bit values for the periodic map2 problems; the others inject particles by 32-bit
    draws and remove them at walls, which 64-bit arithmetic does not reproduce particle by
    particle (charges and counts are whole numbers and must be equal anyway)."""
    if case["kind"] != "map2" or (case["do"] == "cycle" and case["n1"] * case["n2"] > 8192):
        return None
    dev = torch.device("cuda")
    n1, n2 = case["n1"], case["n2"]
    w, phi = _workload(case, seed)
    ps = w.particles[0]
    order = np.argsort(ps.cell, kind="stable") if case["do"] == "handover" else slice(None)
    cell = torch.from_numpy(wl.unpack_cells(ps.cell[order], 2)).to(dev).double()
    t = torch.from_numpy(ps.t[:, order]).to(dev).double()
    v = torch.from_numpy(ps.v[:, order]).to(dev).double()
    k, area, a = _metric(n1, n2, 0.05, dev)
    phi = torch.from_numpy(phi).to(dev)
    if case["do"] != "handover":
        v = _step64((n1, n2), k, phi, cell, t, v, -0.5 * w.dt, -1.0)[2]  # half a step back
    for _ in range(case["steps"]):
        cell, t, v, vv = _step64((n1, n2), k, phi, cell, t, v, w.dt, -1.0)
    if case["do"] == "handover":
        return [None, t, v]
    weight = w.species[0].w
    out = {"charge0": None, "counts": None, "kinetic": 0.5 * weight * float(vv)}
    if case["do"] == "cycle":
        out["phi"], out["field"] = _solve64(n1, n2, area, a, cell, t, weight)
    return out
