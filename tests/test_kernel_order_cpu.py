"""Memory order inside the spreading and interpolation kernels, read from their source (no GPU): what
the lanes write to shared memory together is ordered by a barrier before the lanes stage points over
it or read it.  Shuffles, ballots and reductions order no memory."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2302_00414_gb300", "csrc")
BARRIER = re.compile(r"__sync(warp|threads)\(\)")


@pytest.mark.parametrize("name,function", [
    ("spreadmma.cuh", "spread2d_mma_item"),
    ("spreadmma3.cuh", "k_spread3d_mma"),
    ("spread64.cuh", "spread2d_f64_item"),
    ("spread3d.cuh", "k_spread3d"),
    ("interpco.cuh", "k_interp_co"),
])
def test_barrier_between_clearing_and_staging(name, function):
    """From the last cooperative write of a work item's set-up (the window table, the cleared cells or
    slots) to the first lane that stages a point, the source passes a barrier."""
    text = re.sub(r"//.*", "", open(os.path.join(CSRC, name)).read())
    body = text[re.search(r"\b%s\(const" % function, text).end():]
    stage = re.search(r"if \(lane < (np|mine)\)", body).start()
    writes = [m.end() for m in re.finditer(r"for \(int e = (lane|threadIdx\.x);[^;]*;[^)]*\)[^;]*;", body[:stage])]
    assert writes, "no cooperative write found"
    assert BARRIER.search(body[writes[-1]:stage])
