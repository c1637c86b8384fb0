"""Behind a block that one elected thread of a warp runs, the warp is brought together before it comes to a barrier or elects again:
bar.sync, bar.arrive and elect.sync want all its threads at once, and the elected one may have waited.  Checked on the sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_32114_b200", "csrc")
NEXT = re.compile(r"__syncwarp|aborted\(\)|named_sync|named_arrive|elect_one\(\)|csync\(|__syncthreads|tmem_\w*alloc")


def _statement_end(src, i):
    """The end of the statement that starts at src[i:]."""
    while src[i].isspace():
        i += 1
    if src[i] != "{":
        return src.index(";", i) + 1
    depth = 0
    for j in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        if depth == 0:
            return j + 1
    raise ValueError("unbalanced")


def _block_end(src, i):
    """The end of the block that src[i:] is in."""
    depth = 0
    for j in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        if depth < 0:
            return j
    return len(src)


def loose_ends(src):
    """What follows elected blocks, in the block that they are in (which may be a loop's), without a __syncwarp (or the warp-wide vote in
    aborted()) between."""
    src = re.sub(r"//[^\n]*", "", src)
    bad = []
    for m in re.finditer(r"\bif \((?:\w+ && )?elect_one\(\)\)", src):
        end = _statement_end(src, m.end())
        nxt = NEXT.search(src, end, _block_end(src, end))
        if nxt is None or nxt.group() not in ("__syncwarp", "aborted()"):
            bad.append((src.count("\n", 0, m.start()) + 1, nxt and nxt.group()))
    return bad


@pytest.mark.parametrize("name", sorted(os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*.cu"))))
def test_sources(name):
    assert loose_ends(open(os.path.join(CSRC, name)).read()) == []


def test_the_elected_blocks_are_found():
    src = open(os.path.join(CSRC, "tc_walk.cu")).read()
    assert len(re.findall(r"\bif \((?:\w+ && )?elect_one\(\)\)", src)) == src.count("elect_one()") > 5


@pytest.mark.parametrize("src", ["if (elect_one()) { wait1(a, c); } named_sync(1, 64);", "if (KDA && elect_one()) wait1(a, c);\n named_arrive(1, 64);",
                                 "if (elect_one()) {\n for (;;) { x(); }\n }\n if (elect_one()) y(); __syncwarp();", "{ if (elect_one()) z(); } __syncwarp();"])
def test_planted(src):
    assert len(loose_ends(src)) == 1


def loose_waits(src):
    """Polling waits of the two issuing warps, which the threads of a warp may leave one by one."""
    src = re.sub(r"//[^\n]*", "", src)
    src = src[src.index("if (warp == W_MMA) {"):src.index("warp >= W_OUT")]
    nxt = [NEXT.search(src, m.end(), _block_end(src, m.end())) for m in re.finditer(r"wait1\(", src)]
    assert len(nxt) >= 7
    return [n and n.group() for n in nxt if n is None or n.group() != "__syncwarp"]


def test_the_issuing_warps_wait_together():
    assert loose_waits(open(os.path.join(CSRC, "tc_walk.cu")).read()) == []


@pytest.mark.parametrize("behind,find", [("umma_commit(bar_x);", loose_ends), ("umma_commit(half ? bar_u1 : bar_u0);", loose_ends), ("umma_commit(bar_o);", loose_ends), ("wait1(&full_k[st], ph);", loose_waits),
                                         ("wait1(full_p, c);", loose_waits)])
def test_planted_in_the_kernel(behind, find):
    src = open(os.path.join(CSRC, "tc_walk.cu")).read()
    first = src.index(behind)
    assert find(src[:first] + src[first:].replace("__syncwarp();", "", 1))


# The start states' kernel issues its copies behind a test of the thread index, polls in every thread, and has its barriers and warp-wide
# instructions in the code itself.
ALIGNED = re.compile(r"__syncwarp|__syncthreads|\"bar\.|\b(?:ldsm4t?|stsm\w+|mma_\w+|transpose8x8|put|sync4)\(")


def split_warps(src):
    """Where threads of a warp may part, behind a polling wait or a block for one thread, and what aligned instruction comes next in the source
    if not a __syncwarp or a __syncthreads."""
    src = re.sub(r"//[^\n]*", "", src)
    ends = [src.index(";", m.end()) + 1 for m in re.finditer(r"\bmbar_wait\(", src)]
    ends += [_statement_end(src, m.end()) for m in re.finditer(r"\bif \((?:\(?threadIdx\.x(?: & \d+\))?|tid|lane) (?:==|<) \d+\)", src)]
    bad = []
    for end in ends:
        nxt = ALIGNED.search(src, end)
        if nxt and nxt.group() not in ("__syncwarp", "__syncthreads"):
            bad.append((src.count("\n", 0, end) + 1, nxt.group()))
    return bad


def test_the_start_states_warps_stay_together():
    src = open(os.path.join(CSRC, "tc_span.cu")).read()
    assert src.count("mbar_wait(") == 1 and src.count("fetch(s") == 2   # (what there is to be found)
    assert split_warps(src) == []


@pytest.mark.parametrize("src", ["mbar_wait(a, 0, f);\n}; asm volatile(\"bar.sync 1, 512;\");", "if (lane == 0) x(); asm volatile(\"bar.arrive 2, 512;\");",
                                 "if ((threadIdx.x & 255) == 0) fetch(s);\n ldsm4(w, a);", "if (threadIdx.x == 0)\n for (;;) fetch(s);\n put(h, 1); __syncwarp();",
                                 "if (lane < 16) {\n y();\n } sync4();"])
def test_planted_split(src):
    assert len(split_warps(src)) == 1


@pytest.mark.parametrize("which", [0, 1, 2])
def test_planted_in_the_start_states(which):
    src = open(os.path.join(CSRC, "tc_span.cu")).read().split("__syncwarp();")
    assert len(src) == 4 and len(split_warps("__syncwarp();".join(src[:which + 1]) + "__syncwarp();".join(src[which + 1:]))) == 1


def test_barriers_behind_unequal_work():
    """d = 64: half of a warp stores its columns and lanes run through loops of different length ahead of the barrier of the solving warps."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "fp32_d64.cu")).read())
    assert "if (lane < 16)" in src and "for (int m = c & 16;" in src
    barriers = re.findall(r"(__syncwarp\(\);\s*)?asm volatile\(\"bar\.", src)
    assert barriers and all(barriers)
