"""Bounded waits of the one-CTA and cluster solver kernels for their bulk copies. What goes wrong
without them is undefined on the device, so it is held to the source here, not provoked."""
import os
import re
import struct

import pytest

from paper_1311_2286_gb300 import workloads as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MG = open(os.path.join(ROOT, "paper_1311_2286_gb300", "csrc", "mg.cu")).read()


def kernels():
    """name -> body of every __global__ function of mg.cu that waits for bulk copies."""
    found = {}
    for part in re.split(r"\n__global__ ", MG)[1:]:
        body = part[: part.index("\n}\n")]
        if "bulk_wait(" in body:
            found[re.search(r"(\w+)\(const __grid_constant__", body).group(1)] = body
    return found


def test_barrier_is_initialised_before_any_thread_waits():
    """One thread initialises the mbarrier and starts the copies: a block barrier lies between that
    and the first wait of the other threads."""
    found = kernels()
    assert len(found) >= 3, sorted(found)
    for name, body in found.items():
        between = body[body.index("load.arrive();") : body.index("bulk_wait(")]
        assert "__syncthreads();" in between, name


def test_no_wait_goes_unanswered():
    """A wait that runs out is bounded in time, sets the status the host reads, and is followed by a
    second one before the kernel leaves the memory its copies write."""
    for name, body in kernels().items():
        assert not re.search(r"^\s*bulk_wait\(", body, flags=re.M), name
        assert "= MG_WAIT_RAN_OUT" in body and "(void)bulk_wait(&bar);" in body, name
    wait = MG[MG.index("bool bulk_wait(") :]
    assert "clock64() - start < BULK_WAIT" in wait[: wait.index("\n}\n")]


@pytest.mark.gpu
def test_a_wait_that_ran_out_reaches_the_caller(cpic, tmp_path):
    """The status of such a wait, written into a checkpoint's counters: reported by the diagnostics
    after steps, cleared by the next solve."""
    run = cpic.run_from_workload(wl.langmuir_map2(32, 32, ppc=4), sort_interval=4)
    run.initialize()
    run.step(1)
    d = run.diag()
    path = tmp_path / "state"
    run.checkpoint(str(path))
    run.close()
    data = bytearray(path.read_bytes())
    at = data.find(struct.pack("<d", d["mg_residual"]))  # then ||b||, the cycles and the status
    assert at > 0 and struct.unpack_from("<ii", data, at + 16) == (d["mg_cycles"], 1)
    struct.pack_into("<i", data, at + 20, -1)
    path.write_bytes(data)
    run = cpic.Run.restore(str(path))
    with pytest.raises(cpic.CpicError) as e:
        run.diag()
    assert e.value.status == -5
    run.step(2)
    with pytest.raises(cpic.CpicError) as e:
        run.diag()
    assert e.value.status == -5
    run.solve_field(rtol=1e-10, max_cycles=100)
    assert run.diag()["mg_residual"] <= 1e-10
    run.close()
