"""Rules of the device sources that no run can show."""
import os
import re

import pytest

from paper_2603_06492_gb300.build import CSRC


# kernels that griddepcontrol.wait in a programmatic launch and then read what
# the kernel before them, still running when they became resident, has written
@pytest.mark.parametrize("name", ["simt.cuh", "tc_cosnet.cuh", "sums.cuh"])
def test_no_read_only_loads_in_programmatic_dependents(name):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    assert re.findall(r"__ldg\w*|ld\.global\S*\.nc|__restrict__", text) == []
