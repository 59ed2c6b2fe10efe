"""Device memory of a run: the particles' numbers that make a step's sort cheap take 4 bytes a slot,
and are planned only where a step can number its particles."""
import pytest

from paper_1311_2286_gb300 import workloads as wl


@pytest.fixture(scope="module")
def lib():
    from paper_1311_2286_gb300 import build, cpic

    cpic.load(build.build())
    return cpic


WORKLOADS = {
    "cylinder": (lambda: wl.cylinder(16, 32, npart_per_species=50_000), True),
    "sphere": (lambda: wl.sphere(8, 8, 8, npart_per_species=50_000), True),
    "periodic": (lambda: wl.langmuir_map2(16, 16, ppc=200), True),
    "axisymmetric": (lambda: wl.sphere_axisym(16, 16, npart_per_species=50_000), False),
    "reflecting": (lambda: wl.box_reflect(16, 16, npart=50_000), False),
}


@pytest.mark.parametrize("name", list(WORKLOADS))
def test_numbers_are_planned_where_a_step_can_use_them(lib, name):
    mk, numbers = WORKLOADS[name]
    w = mk()
    sizes = [lib.Run.footprint(lib.config_from_workload(w, sort_interval=k)) for k in (0, 1, 4)]
    cfg = lib.config_from_workload(w)
    slots = sum((int(cfg.capacity[s]) + 31) // 32 * 32 for s in range(cfg.n_species))
    assert sizes[1] == sizes[2]
    if numbers:
        assert 4 * slots <= sizes[1] - sizes[0] < 4 * slots + 256
    else:
        assert sizes[1] == sizes[0]
