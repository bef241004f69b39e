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


def _body(text, head):
    """Source of the function whose definition contains ``head``."""
    start = text.index("\n{", text.index(head))
    return text[start:text.index("\n}", start)]


# what these decide changes the order of sums or the size of a buffer: the shape
# decides, so that results and sizes are the same on every device
@pytest.mark.parametrize("head", ["noble_status simt_launch(", "BwdPlan bwd_plan(", "int simt_tokens_per_thread(",
                                  "WorkLayout work_layout(", "SavedLayout saved_layout("])
def test_summation_orders_do_not_depend_on_the_device(head):
    with open(os.path.join(CSRC, "noble_api.cu")) as f:
        body = _body(f.read(), head)
    assert len(body) > 100 and "num_sms" not in body and "max_clusters" not in body
