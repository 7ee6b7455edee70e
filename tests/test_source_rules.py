"""Rules that the kernels' source keeps and no run can show: the compiler need not
break them on this version."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_03989_gb300", "csrc")


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cuh", ".cu"))))
def test_own_stores_are_not_read_back_by_loads_that_do_not_say_so(name):
    """__ldcg (and ld_state, which is __ldcg) is inline assembly without a "memory"
    clobber: after a plain store to the same address, the store may be dropped or
    delayed past it. The kernels' output pointers (Di, Dk: pixel state, O, dst: node
    state) are read back by plain loads only."""
    with open(os.path.join(CSRC, name)) as f:
        code = re.sub(r"//[^\n]*", "", f.read())
    assert re.findall(r"\b(?:__ldcg|ld_state)\s*\(\s*&?\s*(?:Di|Dk|O|dst)\b[^;]*", code) == []
