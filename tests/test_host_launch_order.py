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


def _pair():
    return _text(os.path.join(CSRC, "sm100_ptx.cuh")), [b for _, n, b in KERNELS if n == "attend_pair_kernel"][0]


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


def _check_order_of_the_paired_kernel(body):
    """The same for the paired kernel, whose CTAs allocate either ahead of the roles or, in the two-CTA form's long launches, in the
    producer's branch, and whose roles wait for the launch before on their own, right before what needs it."""
    one = re.compile(r"if \(!kOwnLate && warp == kProducerWarp\) allocate\(\);\s*tc_fence_before\(\);\s*__syncthreads\(\);")
    late = re.compile(r"auto own_late = \[&\]\(\) \{\s*if \(!kOwnLate\) return;\s*if \(warp == kProducerWarp\) allocate\(\);\s*"
                      r"tc_fence_before\(\);\s*barrier_of\(1, C::kThreads\);")
    early, later = one.search(body), late.search(body)
    assert early and later and len(re.findall(r"\ballocate\(\)", body)) == 2
    cuts = [body.index(t) for t in ("if (layout_ok && warp == kProducerWarp) {", "} else if (layout_ok && warp >= kMmaWarp) {", "} else if (layout_ok) {",
                                    "if constexpr (kSplit) {")]
    assert later.end() < cuts[0] and cuts == sorted(cuts)
    before, producer, issuer, softmax = (body[a:b] for a, b in zip([0] + cuts, cuts))
    assert not re.search(r"tma_load|wait_for_previous|let_next_start", before)
    # the producer: owns, waits, lets the next launch in, loads
    assert len(re.findall(RELEASE, body)) == 1
    order = [producer.index(t) for t in ("own_late();", "if (sq == 0) {", "wait_for_previous();", "let_next_start();", "tma_load")]
    assert order == sorted(order) and producer.count("own_late();") == 1
    assert re.search(r"if \(sq == 0\) \{\s*wait_for_previous\(\);\s*let_next_start\(\);\s*\}", producer)
    # an issuing warp: owns, waits for the launch before, and only then in a wait that has a limit
    order = [issuer.index(t) for t in ("own_late();", "if (tcount[i] == 0) wait_for_previous();", "if (!await(q_full0", "!await(kv_full0", "umma_s<")]
    assert order == sorted(order)
    # the softmax warps: the one that loads queries waits before its first load, all of them before their first S where they own late
    order = [softmax.index(t) for t in ("if (q_armed == 0) wait_for_previous();", "mbar_expect_tx", "tma_load", "own_late();", "mbar_wait(s_full")]
    assert order == sorted(order)
    assert re.search(r"own_late\(\);\s*if \(kOwnLate\) wait_for_previous\(\);", softmax)


def test_the_roles_of_the_paired_kernel_own_and_wait_before_they_load():
    _check_order_of_the_paired_kernel(_pair()[1])


@pytest.mark.parametrize("old,new", [
    ("allocate();\n    tc_fence_before();\n    __syncthreads();", "{}\n    tc_fence_before();\n    __syncthreads();\n    allocate();"),
    ("        barrier_of(1, C::kThreads);\n", ""),
    ("        own_late();\n        uint32_t st_sq", "        uint32_t st_sq"),
    ("                        let_next_start();\n", "                        let_next_start();\n                        own_late();\n"),
    ("if (sq == 0) {\n                        wait_for_previous();", "if (sq == 0) {"),
    ("if (sq == 0) {\n", "if (sq == 1) {\n"),
    ("if (tcount[i] == 0) wait_for_previous();", ""),
    ("if (q_armed == 0) wait_for_previous();", ""),
    ("if (kOwnLate) wait_for_previous();", ""),
    ("auto own_late = [&]() {", "let_next_start();\n    auto own_late = [&]() {"),
])
def test_the_check_of_the_roles_order_rejects(old, new):
    body = _pair()[1]
    assert body.count(old) == 1
    with pytest.raises((AssertionError, ValueError)):
        _check_order_of_the_paired_kernel(body.replace(old, new))


def test_a_producer_that_owns_its_columns_behind_the_release_is_rejected():
    body = _pair()[1]
    moved = body.replace("        own_late();\n        uint32_t st_sq", "        uint32_t st_sq")
    moved = moved.replace("let_next_start();\n", "let_next_start();\n                        own_late();\n")
    assert moved != body and moved.count("own_late();") == body.count("own_late();")
    with pytest.raises(AssertionError):
        _check_order_of_the_paired_kernel(moved)


def test_the_producer_of_the_paired_kernel_allocates_as_a_whole_warp():
    """tcgen05.alloc is an aligned instruction, and loops of unequal length or a branch of one lane come before it."""
    body = [b for _, n, b in KERNELS if n == "attend_pair_kernel"][0]
    assert body.count("tcgen05.alloc") == 1
    assert re.search(r"__syncwarp\(\);\s*asm volatile\(\"tcgen05\.alloc", body)


def _check_end_of_a_launch_that_gave_up(header, body):
    """The issuing warps of the paired kernel issue nothing more once a wait of theirs has given up -- their commits are what the other
    roles take for landed data and free stages -- and what is under way then ends before memory is given back."""
    wait = re.search(r"bool warp_wait_lean\(.*?\n}", header, flags=re.S).group(0)
    assert wait.count("__all_sync(0xffffffffu, mbar_try_wait(bar, parity))") == 2 and "__any_sync(0xffffffffu, *abort_flag)" in wait
    assert wait.count("return true;") == 2 and re.search(r"report\([^;]*;\s*return false;", wait)
    role, end = body[: body.rindex("dealloc")].rsplit("if (layout_ok && *abort_flag) {", 1)
    issuer = role[role.index("warp >= kMmaWarp"):]
    issuer = issuer[: issuer.index("stopped:")]
    assert body.count("warp_wait_lean(") == issuer.count("return warp_wait_lean(") == 1
    for call in ("await", "issue_pv"):
        uses = re.findall(r"(\S*)\b%s\([^;]*;" % call, issuer)
        tails = re.findall(r"\b%s\([^;]*\) (goto stopped|return false);" % call, issuer)
        assert len(uses) == len(tails) >= 3 and all(u.endswith("!") for u in uses)
    assert len(re.findall(r"umma_(?:s|pv|commit_elected)\b[^;]*;", role)) == 4 == len(re.findall(r"umma_(?:s|pv|commit_elected)\b[^;]*;", issuer))
    assert re.search(r"stopped:\s*if \(!owned\) own_late\(\);\s*\}", role)
    assert re.search(r"__syncthreads\(\);\s*$", role)           # all roles have stopped
    assert re.search(r"if \(!ok\) report\([^;]*;\s*bars->issued = sq;", role)
    assert re.search(r"for \(uint32_t q = un; q < q_armed; \+\+q\)", role)
    assert re.search(r"bars->issued.*until\(kv_full0.*umma_commit_elected\(drained\);\s*until\(drained.*__syncthreads\(\);\s*\}\s*if", end, flags=re.S)


def test_a_launch_that_gave_up_issues_nothing_more_and_ends_its_copies():
    _check_end_of_a_launch_that_gave_up(*_pair())


@pytest.mark.parametrize("old,new", [
    ("!await(kv_full0 + 8 * stage, use & 1u)) goto stopped;", "!await(kv_full0 + 8 * stage, use & 1u)) tc_fence_after();"),
    ("if (!await(q_full0 + 16 * g + 8 * q_half[i], (q_split ? u >> 1 : u) & 1u)) goto stopped;",
     "await(q_full0 + 16 * g + 8 * q_half[i], (q_split ? u >> 1 : u) & 1u);"),
    ("if (s_first && pv_live[i] && !issue_pv(i)) goto stopped;", "if (s_first && pv_live[i]) issue_pv(i);"),
    ("if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;", "if (mbar_try_wait(bar, parity)) return true;"),
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
