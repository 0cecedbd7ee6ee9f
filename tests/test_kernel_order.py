"""Orders inside the kernels that no run shows to be wrong until it hangs, checked on the source text."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_01890_b200", "csrc")


def kernels():
    """(file:kernel, body) of every __global__ function, comments taken out."""
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^{;]*?(\w+)\(", re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", lambda b: " " * len(b.group()), text)):
            depth, start = 0, text.index("{", m.end())
            for end in range(start, len(text)):
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                if depth == 0:
                    break
            found.append(("%s:%s" % (os.path.basename(path), m.group(1)), text[start:end]))
    return found


def test_kernels_are_found():
    names = {n.split(":")[1] for n, _ in kernels()}
    assert {"tc_flash_kernel", "tc_align_link_kernel", "tc_project_kernel", "tc_project_narrow_kernel", "decode_merge_kernel"} <= names


@pytest.mark.parametrize("body", [pytest.param(b, id=n) for n, b in kernels() if "tmem_alloc(" in b])
def test_successors_are_released_after_the_tensor_memory_is_held(body):
    """A released successor may take all of an SM's tensor memory and wait for this kernel: a CTA of this kernel without its columns
    would then wait for the successor, without a limit."""
    if "chain_release()" not in body:
        return
    released = body.index("chain_release()")
    barrier = body.index("__syncthreads()", body.index("tmem_alloc("))
    assert released > barrier, "chain_release() comes before the barrier behind tmem_alloc()"


WAITING = [(n, b) for n, b in kernels() if "chain_release()" in b or "chain_wait()" in b]


@pytest.mark.parametrize("body", [pytest.param(b, id=n) for n, b in WAITING])
def test_kernels_of_a_chain_wait_whatever_their_arguments(body):
    """What earlier kernels wrote is visible to a kernel behind its own wait only: one wait, at the top level of the kernel."""
    assert len(re.findall(r"chain_wait\(\)", body)) == 1
    at = body.index("chain_wait()")
    assert body[:at].count("{") - body[:at].count("}") == 1, "the wait is inside a block"
    assert body[:at].rstrip()[-1] in ";}", "the wait hangs on a condition"


@pytest.mark.parametrize("name,inputs", [("pack_lowrank_kernel", ("jobs.",)), ("tc_align_kernel", ("p.w", "p.b", "planes")),
                                         ("tc_align_link_kernel", ("p.w1", "p.b1", "p.w2", "p.b2"))])
def test_prefill_kernels_wait_before_they_read(name, inputs):
    """Q', K' and the weights as well: the kernel right in front of the call may have written them."""
    body = next(b for n, b in WAITING if n.endswith(":" + name))
    assert not [x for x in inputs if x in body[:body.index("chain_wait()")]]
