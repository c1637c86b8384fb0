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


# ... and by way of copies, helpers, casts and pointers made from a parameter
ACCESS = (r"\b(?:bulk_load|tma_load_4d|prefetch_l2|__ldcs|__ldg|__ldcg|__stcs|load4|ld4|load_tile|load_gates|issue_tiles|fetch|atomic\w+)\s*\("
          r"|reinterpret_cast<[^>]*\*>\(p\.\w+[^)]*\)\s*\[|(?<=[=(,?:])\s*\*\s*\(?(?:p|sb)\.|(?<![\w.])(?:src|dst|phi|rec|img|gp|my_len)\s*\[")


def accesses(before):
    """Accesses in the code that runs ahead of the wait: all but the bodies of lambdas, which are called later or found by name."""
    flat = re.sub(r"auto \w+ = \[&\]\([^)]*\) \{(?:[^{}]|\{[^{}]*\})*\};", "", before)
    return re.findall(ACCESS, flat)


@pytest.mark.parametrize("file,kernel,body", list(_kernels()), ids=lambda x: x if isinstance(x, str) and len(x) < 30 else "")
def test_no_copy_or_pointer_is_followed_before_the_wait(file, kernel, body):
    assert accesses(body[body.index("{"):body.index("griddepcontrol.wait")]) == [], f"{kernel} in {file}"


@pytest.mark.parametrize("early", ["bulk_load(sm, rec + kStepT, kTriB, &full[0]);", "tma_load_4d(sm, &map_k, &full[0], 0, j, t0, 0);", "fetch(1);",
                                   "load_tile(b, h);", "const float x = src[lane];", "vv = load4(reinterpret_cast<const In*>(p.v) + nj);",
                                   "len = *(p.seq_len + n);", "len = *p.seq_len;", "sk[0] = to_f32(reinterpret_cast<const In*>(p.k)[qk]);",
                                   "h = __ldcs(reinterpret_cast<const float4*>(p.h_in + base));", "issue_tiles(gm, 0);", "q = ld4(p.g + off);"])
def test_planted_access_before_the_wait(early):
    for _, kernel, body in _kernels():
        at = body.index("asm volatile(\"griddepcontrol.wait")
        assert accesses(body[body.index("{"):at] + early), kernel


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


def test_outputs_are_not_sent_past_l2():
    """They are what the caller's next kernel reads."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "tc_walk.cu")).read())
    assert "orow + " in src and not re.search(r"__st(?:cs|cg|wt)\(|st\.global\.(?:cs|L1::no_allocate)|L2::cache_hint", src)


def _copying_kernels():
    """Every kernel that copies in bulk, its body."""
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(f).read())
        for part in src.split("__global__")[1:]:
            name, body = re.search(r"(\w+_kernel)\s*\(", part), part[part.index("{"):part.index("\n}")]
            if re.search(r"\b(?:bulk_load|tma_load_4d)\(", body):
                yield name.group(1), body


def unreported(kernels, header):
    """Kernels that copy in bulk and neither report a wait that ran out, themselves or by the header's helper, nor let their copies land then."""
    pause = r"report_status\([^;]*HA_LA_ERR_TIMEOUT\);\s*(?:ptx::)?settle_copies\(\);"
    helper = re.search(r"void report_timeout\([^)]*\) \{\s*" + pause, re.sub(r"//[^\n]*", "", header))
    return [k for k, body in kernels if not re.search(pause, body) and not (helper and "report_timeout(" in body)]


def test_kernels_that_copy_report_a_wait_that_ran_out():
    header = open(os.path.join(CSRC, "fp32_common.cuh")).read()
    kernels = list(_copying_kernels())
    assert {k for k, _ in kernels} == {"tc_tp_kernel", "tc_kda_kernel", "tc_walk_kernel", "span_fix_kernel", "fp32_walk_kernel", "fp32_walk64_kernel"}
    assert unreported(kernels, header) == []
    assert unreported(kernels, header.replace("ptx::settle_copies();", "")) == ["fp32_walk64_kernel"]
    for k, body in kernels:                                # (planted: nobody reports)
        assert unreported([(k, re.sub(r"report_\w+\(", "x(", body))], header) == [k]
