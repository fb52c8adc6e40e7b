"""Hand-overs through shared memory inside a warp: a barrier stands between the store and the load."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1905_07440_gb300", "csrc")


def test_reflector_entries_pass_a_warp_barrier():
    """Lane j of a panel warp stores its row's entries in ps->a and every lane reads one: shuffles in between
    move registers and order no memory."""
    code = re.sub(r"//.*", "", open(os.path.join(CSRC, "hq_panel.cuh")).read())
    store = code.index("ps->a[warp][i] = ")
    load = code.index("= ps->a[warp][", store + 1)
    assert "__syncwarp()" in code[store:load]
