"""Launch overlap in the CUDA sources, checked on the text: the order of its instructions, where what it guards against is a hang,
which no test may provoke on a GPU, and the loads behind them, where it is a compiler's licence."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_16047_b200", "csrc")


def _kernels():
    """(file, name, body) of every __global__ function; comments removed."""
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
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
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
    assert not re.search(r"__ld(g|cs|ca|cg|lu|cv)\s*\(|ld\.global\.nc", text)
    for m in re.finditer(r"__global__", text):
        assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", text[m.end():text.index("{", m.end())])
