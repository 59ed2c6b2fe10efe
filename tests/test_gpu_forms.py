"""Layouts of the cluster solver that the grids elsewhere in this suite do not reach: levels too large
for a thread's registers, two and three split levels with closed and periodic second axes, one CTA,
the shortest rows. The layout is held to what the launch shows, where a profiler is at hand, and the
solution to the oracle's operator at the tolerance whose status the call returned."""
import json
import os

import numpy as np
import pytest

from oracle import geometry, poisson
from paper_1311_2286_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

P, Dr, Ne = 0, 1, 2
PP, PA, PR = 0, 1, 2


def rectangle(n1, n2):
    """Square cells."""
    x, y = np.meshgrid(np.arange(n1 + 1.0), np.arange(n2 + 1.0), indexing="xy")
    return np.stack([x, y], axis=-1) / 16.0


def launches(torch, fn, path):
    """(kernel name, blocks) of every launch of fn; empty where nothing can be recorded."""
    from torch.profiler import ProfilerActivity, profile

    with profile(activities=[ProfilerActivity.CUDA]) as p:
        fn()
        torch.cuda.synchronize()
    p.export_chrome_trace(str(path))
    events = json.load(open(path))["traceEvents"]
    os.remove(path)
    return [(e["name"], e["args"]["grid"][0]) for e in events if e.get("cat") == "kernel"]


# grid, boundaries, Omega = r, CTAs of the launch
LAYOUTS = {
    "one_cta": ((4, 32), [Dr, Dr, P, P], False, 1),
    "short_rows": ((4, 64), [Dr, Ne, Dr, Ne], False, 8),
    "two_ctas": ((24, 32), [Dr, Dr, P, P], False, 2),
    "large_legs": ((288, 32), [Dr, Dr, P, P], False, 4),
    "large_legs_closed": ((288, 32), [Dr, Ne, Dr, Ne], False, 4),
    "large_legs_periodic": ((272, 32), [P] * 4, False, 4),
    "two_split_closed": ((16, 704), [Ne, Dr, Dr, Dr], False, 16),
    "two_split_omega_r": ((128, 128), [Dr, Dr, Ne, Ne], True, 8),
    "two_split_periodic": ((32, 416), [P] * 4, False, 8),
    "three_split": ((32, 1536), [Dr, Dr, P, P], False, 16),
    "three_split_wide": ((128, 384), [Dr, Dr, P, P], False, 16),
    "three_split_periodic": ((64, 768), [P] * 4, False, 16),
}


@pytest.mark.parametrize("name", list(LAYOUTS))
def test_cluster_layouts(cpic, name, monkeypatch, tmp_path):
    torch = pytest.importorskip("torch")
    monkeypatch.delenv("CPIC_NO_CLUSTER_SOLVER", raising=False)
    n, bc, axisym, ctas = LAYOUTS[name]
    X = wl.sphere_axisym_vertices(*n, 1.0, 10.0) if axisym else rectangle(*n)
    bv = [v if b == Dr else 0.0 for v, b in zip((-2.5, 0.0, 0.7, -0.4), bc)]
    periodic = [bc[0] == P, bc[2] == P]
    g = geometry.build_geometry(X, periodic, axisym=axisym)
    M, bbc = poisson.assemble(g, bc, bv)
    npart = 5000
    rng = np.random.default_rng(21)
    idx = np.stack([rng.integers(0, n[a], npart) for a in range(2)])
    t = rng.random((2, npart)).astype(np.float32)
    pbc = [PP if b == P else (PR if axisym else PA) for b in bc]
    run = cpic.Run(cpic.make_config(2, n, bc, bv, pbc, 0.1, [(-1.0, 1.0, 1e-3, npart)], background=0.3,
                                    axisymmetric=axisym))
    run.set_map_vertices(X)
    run.load_particles(0, wl.pack_cells(idx), t, np.zeros((3, npart), np.float32))
    run.deposit()
    seen = launches(torch, lambda: run.solve_field(rtol=1e-10, max_cycles=100), tmp_path / "trace.json")
    cluster = [blocks for kernel, blocks in seen if "mg_cluster_kernel" in kernel]
    assert not seen or cluster == [ctas]
    run.set_phi(np.zeros((n[1], n[0])))
    cycles, res = run.solve_field(rtol=1e-10, max_cycles=100)  # raises unless the status is OK
    Q = poisson.charge_in_cells(g, [run.charge(0)], [-1e-3], 0.3)
    assert 0 < cycles and res <= 1e-10
    # the device's FP64 residual and the oracle's differ by their roundings
    assert poisson.residual_norm(M, bbc, g, Q, run.phi(), bc) <= 1.01e-10
    run.close()
