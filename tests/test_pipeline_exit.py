"""A block must not end with copies still landing in its shared memory.  Whether
they can is a property of the exit path after an expired wait, which no test
can take on a GPU without the fault it would show; so the sources are read: every
producer of bulk or TMA copies waits for the last ones it issued whatever made
its loop end, and only the choice of the barrier may depend on that."""
import os
import re

import paper_2412_18553_gb300

CSRC = os.path.join(os.path.dirname(paper_2412_18553_gb300.__file__), "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_energy_producer_waits_for_its_last_copies_on_every_exit():
    body = _code("energy_tc.cu").split("ptx::bulk_load", 1)[1].split("compute warps", 1)[0]
    loop_end = body.index("issued = true;")
    waits = re.findall(r"if \(([^;{}]*)\) ptx::mbar_wait\(&full\[b\]", body[loop_end:].split("} else {")[0])
    assert len(waits) == 1
    assert "issued" in waits[0] and not re.search(r"\bok\b|abort_flag", waits[0]), waits[0]


def test_contraction_producers_wait_for_every_pending_stage():
    for name in ("tc_path.cu", "view_tc.cu"):
        code = _code(name)
        tail = code.split("if (pending[s] < 0) continue;", 1)[1].split("} else if (warp == 1)", 1)[0]
        assert re.search(r"ptx::mbar_wait\(&empty\[s\]", tail) and re.search(r"ptx::mbar_wait\(&full\[s\]", tail), name
        assert "pause_ns" in tail, name
