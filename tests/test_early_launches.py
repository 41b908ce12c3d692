"""What a kernel that is launched while the one before it drains has to keep to, read off the sources: a mistake in it would be a race
or two kernels that wait for each other, which no run is to show."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_04405_b200", "csrc")
WAIT = r"pdl_wait\(\)|griddepcontrol\.wait"
RELEASE, ALLOC = r"pdl_release\(\)|griddepcontrol\.launch_dependents", r"tcgen05\.alloc"
BLOCK_BARRIER = r"__syncthreads\(\)|barrier\.cluster\.wait"


def _kernels():
    """{name: (parameters, body)} of every kernel; comments taken out."""
    found = {}
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__\b[^;{]*\{", src):
            head = m.group(0)[:m.group(0).rindex(")")]
            depth, start = 1, len(head)
            while depth:                                     # (back to the parenthesis that opens the parameters)
                start -= 1
                depth += {")": 1, "(": -1}.get(head[start], 0)
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
            name = re.search(r"(\w+)(?:<[^()]*>)?\s*$", head[:start]).group(1)
            found[f + ":" + name] = (head[start + 1:], src[m.end():end])
    return found


KERNELS = _kernels()
EARLY = sorted(k for k, (_, body) in KERNELS.items() if re.search(RELEASE, body))


def test_the_kernels_are_found():
    names = {k.split(":")[1] for k in EARLY}
    assert {"dots_kernel", "append_kernel", "encode_simple_kernel", "encode_tc_kernel", "fit_project_tc_kernel", "fit_gather_tc_kernel",
            "fit_sweep_kernel", "fit_sum_parts_kernel", "fit_rows_kernel", "fit_finish_kernel", "bpc_decode_kernel"} <= names


@pytest.mark.parametrize("kernel", [k for k in EARLY if re.search(ALLOC, KERNELS[k][1])])
def test_tensor_memory_is_held_before_the_next_kernel_may_start(kernel):
    """A kernel that allocates ahead of its wait keeps the columns until the one before it is through.  If that one may still have to
    allocate, on an SM where both have room, each waits for the other."""
    body = KERNELS[kernel][1]
    alloc = re.search(ALLOC, body).end()
    barrier = alloc + re.search(BLOCK_BARRIER, body[alloc:]).end()
    assert not re.search(RELEASE, body[:barrier])


@pytest.mark.parametrize("kernel", EARLY)
def test_nothing_is_written_to_global_memory_ahead_of_the_wait(kernel):
    """What lies there may be in use by the kernel before, or by the one before that."""
    params, body = KERNELS[kernel]
    body = re.sub(r"\{\s*pdl_wait\(\);[^{}]*\breturn;\s*\}", "return;", body)   # (a block that leaves behind a wait of its own)
    ahead = body[:re.search(WAIT, body).start()]
    for f in re.findall(r"\*\s*(?:__restrict__\s+)?(\w+)", ",".join(p for p in params.split(",") if "const" not in p)):
        names = {f}
        for m in re.finditer(r"\*\s*(\w+)\s*=([^;]*);", ahead):
            if names & set(re.findall(r"\w+", m.group(2))):
                names.add(m.group(1))
        for name in names:
            assert not re.search(r"(?:\b%s|\(%s\))\s*\[[^;=]*\]\s*[-+|&]?=(?!=)" % (name, name), ahead), name


@pytest.mark.parametrize("kernel", EARLY)
def test_what_the_kernel_before_writes_is_read_coherently(kernel):
    """`const` with `__restrict__` allows loads through the read-only path and ahead of the wait: both need memory that nobody writes while the
    kernel is resident, and it is resident while the one before still writes.  The directions and lengths of a fit are older."""
    params, body = KERNELS[kernel]
    older = {"v_star", "unit_lens"} if kernel.startswith("fit_block.cu") else set()
    assert set(re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params)) <= older
    assert "__ldg" not in body


def test_no_load_through_the_read_only_path():
    """(the same for loads written out: the codes of a step may be those of the kernel before)"""
    for f in os.listdir(CSRC):
        assert "ld.global.nc" not in open(os.path.join(CSRC, f)).read(), f


@pytest.mark.parametrize("kernel", EARLY)
def test_no_block_leaves_ahead_of_the_wait(kernel):
    """A kernel whose blocks all leave ahead of their wait (lengths of zero) is over before the one before it, and what follows would start
    beside that one."""
    body = KERNELS[kernel][1]
    ahead = body[:re.search(r"\n  (?:%s|asm volatile\(\"griddepcontrol\.wait)" % WAIT.split("|")[0], body).start()]
    for m in re.finditer(r"\breturn;", ahead):
        statement = ahead[max(ahead.rfind("if (", 0, m.start()), 0):m.start()]
        assert re.search(WAIT, statement), statement
