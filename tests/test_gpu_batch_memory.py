"""A planned batch keeps no host copy of its uploaded task graph."""
import ctypes
import gc

import numpy as np
import pytest

import schur_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class MallInfo(ctypes.Structure):
    _fields_ = [(k, ctypes.c_size_t) for k in ("arena", "ordblks", "smblks", "hblks", "hblkhd", "usmblks",
                                               "fsmblks", "uordblks", "fordblks", "keepcost")]


def heap_in_use():
    libc = ctypes.CDLL(None)
    if not hasattr(libc, "mallinfo2"):
        pytest.skip("needs glibc's mallinfo2")
    libc.mallinfo2.restype = MallInfo
    i = libc.mallinfo2()
    return i.uordblks + i.hblkhd


@pytest.fixture(scope="module")
def gbr():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1905_04975_gb300 as g
    g.load()
    return g


def test_plan_keeps_no_image(gbr):
    S, Q, sel = si.reorder_problem(400, 5, select_frac=0.4)

    def plan():
        Sd = [gbr.to_device(S) for _ in range(40)]
        Qd = [gbr.to_device(Q) for _ in range(40)]
        return gbr.Batch(Sd, Qd, [sel] * 40, window=16, chain=8)

    plan().run()  # pools, streams and the library's first allocations
    gc.collect()
    before = heap_in_use()
    b = plan()
    grown = heap_in_use() - before
    tasks = b.run().stats.tasks
    # the image holds at least 24 bytes a task (task, two counters); what a plan
    # keeps on the host otherwise (selections, block patterns, plan summaries)
    # is some KB a form
    assert tasks > 100000
    assert grown < 24 * tasks / 4, (grown, tasks)
