"""What a kernel owes the ones around it, checked on the sources, without a GPU.

Kernels that are launched as programmatic dependents may run before the kernel ahead of them in the stream has written
anything, so each has to execute griddepcontrol.wait before its first access to what another kernel writes: the plan kernel's
tables above all, which lie in workspace memory that holds anything until then.  And a kernel in which a bounded wait ran out
lets its own copies land before it gives its shared memory back."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_32114_b200", "csrc")
TABLES = r"\b(?:seq_order|seq_tok0|seq_len|seq_chunk0|chunk_seq|chunk_tok0|chunk_len|cu)\s*\[|\*my_len"
INPUTS = r"\bp\.(?:q|k|v|g|beta|h0|h_in|o|hT|h_out|rec)\s*\["


def _kernels():
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(f).read())
        for part in src.split("__global__")[1:]:
            name = re.search(r"(\w+_kernel)\s*\(", part)
            if name and "griddepcontrol.wait" in part:
                yield os.path.basename(f), name.group(1), part


def test_the_dependent_kernels_are_found():
    names = {k for _, k, _ in _kernels()}
    assert {"plan_kernel", "tc_tp_kernel", "tc_kda_kernel", "tc_walk_kernel", "span_fix_kernel", "fp32_prep_kernel",
            "fp32_walk_kernel", "decode_kernel"} <= names


@pytest.mark.parametrize("file,kernel,body", list(_kernels()), ids=lambda x: x if isinstance(x, str) and len(x) < 30 else "")
def test_nothing_is_read_before_the_wait(file, kernel, body):
    before = body[:body.index("griddepcontrol.wait")]
    assert re.findall(TABLES, before) == [] and re.findall(INPUTS, before) == [], f"{kernel} in {file}"


def test_a_kernel_that_gave_up_waiting_lets_its_copies_land():
    found = 0
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(f).read())
        for m in re.finditer(r"report_status\([^;]*HA_LA_ERR_TIMEOUT\);", src):
            assert src[m.end():].split("}")[0].strip() == "settle_copies();", os.path.basename(f)
            found += 1
    assert found == 5                                      # every kernel that copies in bulk


def test_that_pause_is_by_the_clock():
    """nanosleep may return at once, so the pause has to be measured, and bounded should the clock stand still."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "tc_ptx.cuh")).read())
    body = src[src.index("void settle_copies()"):].split("\n}")[0]
    assert "%globaltimer" in src and re.search(r"for \(int i = 0; i < \d+ && global_ns\(\) - t0 < \d+;", body)
