"""The debug checks cover every device index array of a handle: each array of DevGraph is read
in debug.cu, but the bit-packed rows (values, no indices) and the resident kernels' copy of
arrays that are checked one by one."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_10424_gb300", "csrc")


def test_every_index_array_is_checked():
    with open(os.path.join(CSRC, "ldpc_internal.h")) as f:
        body = re.search(r"struct DevGraph \{(.*?)\n\};", f.read(), re.S).group(1)
    arrays = re.findall(r"u?int(?:8|16|32)_t\* (\w+)", body)
    assert {"row_ptr", "ell_col", "row_slot", "col_k"} <= set(arrays)
    with open(os.path.join(CSRC, "debug.cu")) as f:
        checked = set(re.findall(r"\bg\.(\w+)", f.read()))
    assert set(arrays) - checked == {"packed", "idx_blob"}
