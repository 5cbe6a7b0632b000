"""The warps of the helicity-shared adjoint (no GPU needed).

* A set of lanes that take part in a warp-wide operation is formed with a
  ballot where all of them arrive; which lanes happen to run together after a
  branch (__activemask) is no such set: a shuffle partner outside it gives an
  undefined value, a group split in two has two leaders.
* The momentum and propagator adjoints of four consecutive items are summed
  before they are added, so these agree in type, momentum entries and
  propagator; the generator refuses a table in which they do not.
"""
import glob
import os
import re

import pytest

from paper_2106_12631_gb300 import build as B
from paper_2106_12631_gb300.gen import procgen


def test_no_warp_operation_on_an_accidental_set_of_lanes():
    files = [f for ext in ("cu", "cuh", "h") for f in glob.glob(os.path.join(B.CSRC, "**", "*." + ext), recursive=True)]
    assert files
    for f in files:
        code = re.sub(r"//[^\n]*", "", open(f).read())
        assert "__activemask" not in code, f


@pytest.mark.parametrize("pid", procgen.GRAD_PROCS)
def test_quads_of_adjoint_items_agree(pid, monkeypatch):
    seen = []
    check = procgen.check_adjoint_quads
    monkeypatch.setattr(procgen, "check_adjoint_quads", lambda items, starts: (seen.append((items, starts)), check(items, starts)))
    procgen.generate(pid)
    (items, starts), = seen
    assert starts[0] == 2 * procgen.Process(procgen.PROCS[pid]).n and starts[-1] == len(items)
    # a quad whose last item belongs to another current, or with another momentum entry
    i = starts[0]
    other = next(it for it in items[i:] if it[0] != items[i][0])
    for wrong in (other, items[i + 3][:7] + (items[i + 3][7] + 1,) + items[i + 3][8:]):
        with pytest.raises(ValueError):
            check(items[:i + 3] + [wrong] + items[i + 4:], starts)
    with pytest.raises(ValueError):
        check(items, starts[:1] + [starts[0] + 2] + starts[1:])
