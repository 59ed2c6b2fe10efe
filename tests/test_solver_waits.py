"""Bounded waits of the one-CTA and cluster solver kernels for their bulk copies. What goes wrong
without them is undefined on the device, so it is held to the source here, not provoked."""
import os
import re

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
