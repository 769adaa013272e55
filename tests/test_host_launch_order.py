"""Launch overlap and the end of launches that gave up, checked on the text of the CUDA sources: the order of their instructions,
where what it guards against is a hang or a copy into shared memory that has a new owner, which no test may provoke on a GPU, and
the loads behind them, where it is a compiler's licence."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_16047_b200", "csrc")


def _text(path):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)


def _kernels():
    """(file, name, body) of every __global__ function; comments removed."""
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = _text(path)
        for m in re.finditer(r"__global__", text):
            start = text.index("{", m.end())
            name = re.findall(r"(\w+)\s*\(", text[m.end():start])
            depth, end = 0, start
            for end in range(start, len(text)):
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                if depth == 0:
                    break
            found.append((os.path.basename(path), [n for n in name if n.endswith("kernel")][0], text[start:end]))
    return found


KERNELS = _kernels()
RELEASE = r"launch_dependents|overlap_with_previous\s*\(|let_next_start\s*\("
WAIT = r"griddepcontrol\.wait|overlap_with_previous\s*\(|wait_for_previous\s*\("


def test_kernels_are_found():
    assert {"attend_pair_kernel", "attend_mid_kernel", "attend_small_kernel", "append_kernel"} <= {n for _, n, _ in KERNELS}


@pytest.mark.parametrize("name,body", [(n, b) for _, n, b in KERNELS], ids=[n for _, n, _ in KERNELS])
def test_the_next_launch_is_let_in_after_the_wait_and_after_the_tensor_memory_is_owned(name, body):
    """A CTA of the next launch may allocate tensor memory as soon as it is let in, and then waits for this launch to end while
    it holds it.  A CTA of this launch that has not allocated yet would wait for it in turn: every CTA allocates, and
    synchronises on that, before any of its warps lets the next launch in.  And a launch that lets the next one in before its
    own wait would let that one run beside the launch before this one."""
    release = re.search(RELEASE, body)
    if not release:
        return
    wait = re.search(WAIT, body)
    assert wait and wait.start() <= release.start()
    alloc = re.search(r"tcgen05\.alloc", body)
    if alloc:
        owned = re.search(r"__syncthreads\s*\(", body[alloc.end():])
        assert owned and release.start() > alloc.end() + owned.start()


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_no_load_promises_that_its_data_is_read_only(path):
    """A kernel is alive while the one before it still writes, so no load may go by the read-only path, which promises that the
    data does not change and lets the compiler move the load above the wait."""
    text = _text(path)
    assert not re.search(r"__ld(g|cs|ca|cg|lu|cv)\s*\(|ld\.global\.nc", text)
    for m in re.finditer(r"__global__", text):
        assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", text[m.end():text.index("{", m.end())])


def test_the_producer_of_the_paired_kernel_allocates_as_a_whole_warp():
    """tcgen05.alloc is an aligned instruction, and loops of unequal length or a branch of one lane come before it."""
    body = [b for _, n, b in KERNELS if n == "attend_pair_kernel"][0]
    assert body.count("tcgen05.alloc") == 1
    assert re.search(r"__syncwarp\(\);\s*asm volatile\(\"tcgen05\.alloc", body)


def _check_end_of_a_launch_that_gave_up(header, body):
    """The issuing warps of the paired kernel issue nothing more once a wait of theirs has given up -- their commits are what the other
    roles take for landed data and free stages -- and what is under way then ends before memory is given back."""
    blocks = [m.group(0) for m in re.finditer(r"asm volatile\((?:[^;]|;(?!\n\s*(?:\}|else)))*?elect\.sync _\|e.*?\"memory\"\);", header, flags=re.S)]
    assert len(blocks) == 4                                    # a commit, S with 64 and with 128 channels, P V
    for block in blocks:
        assert re.search(r"elect\.sync _\|e, 0xffffffff;\\n\"\s*\"setp\.ne\.and\.u32 e, %\d+, 0, e;", block) and "(uint32_t)go" in block
        assert all(p for p in re.findall(r"(@\w+ )?tcgen05\.(?:mma|commit)", block))
    assert re.search(r"bool wait_through\([^}]*report\([^;]*;\s*return false;", header)
    assert re.search(r"if \(go\) go = wait_through\(", body) and body.count("wait_through(") == 1
    role, end = body[: body.rindex("dealloc")].rsplit("if (layout_ok && *abort_flag) {", 1)
    issued = re.findall(r"umma_(?:s|pv|commit_elected)\b[^;]*;", role)
    assert len(issued) == 4 and all(re.search(r", go\);", call) for call in issued)
    assert re.search(r"__syncthreads\(\);\s*$", role)           # all roles have stopped
    assert re.search(r"if \(!ok\) report\([^;]*;\s*bars->issued = sq;", role)
    assert re.search(r"for \(uint32_t q = un; q < q_armed; \+\+q\)", role)
    assert re.search(r"bars->issued.*until\(kv_full0.*umma_commit_elected\(drained, true\);\s*until\(drained.*__syncthreads\(\);\s*\}\s*if", end, flags=re.S)


def _pair():
    return _text(os.path.join(CSRC, "sm100_ptx.cuh")), [b for _, n, b in KERNELS if n == "attend_pair_kernel"][0]


def test_a_launch_that_gave_up_issues_nothing_more_and_ends_its_copies():
    _check_end_of_a_launch_that_gave_up(*_pair())


@pytest.mark.parametrize("old,new", [
    ("if (go) go = wait_through(", "wait_through("),                            # products behind a wait that gave up
    ("s_full0 + 16 * g + 8 * buf, go);", "s_full0 + 16 * g + 8 * buf, true);"),
    ("umma_commit_elected(empty, go);", "umma_commit_elected(empty, true);"),
    ('"setp.ne.and.u32 e, %11, 0, e;\\n"', ""),
    ('"@r tcgen05.commit', '"tcgen05.commit'),
    ("report(status, code, abort_flag);\n            return false;", "report(status, code, abort_flag);\n            break;"),
    ("if (!ok) report(status, kStatusTmaTimeout, abort_flag);\n            bars->issued = sq;",
     "if (!ok) { report(status, kStatusTmaTimeout, abort_flag); bars->issued = sq; }"),
    ("q = un; q < q_armed", "q = un + 1; q < q_armed"),
    ("            until(drained, 0u);\n        }\n        __syncthreads();", "            until(drained, 0u);\n        }"),
    ("    __syncthreads();\n    if (layout_ok && *abort_flag) {", "    if (layout_ok && *abort_flag) {"),
])
def test_the_check_of_launches_that_gave_up_rejects(old, new):
    header, body = _pair()
    assert (old in header) != (old in body)
    with pytest.raises((AssertionError, ValueError)):
        _check_end_of_a_launch_that_gave_up(header.replace(old, new), body.replace(old, new))
