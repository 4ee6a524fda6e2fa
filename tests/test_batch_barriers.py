"""Batched kernels walk work items, several of one member to a block, and
stage_member synchronises only where the member changes.  A body that shares
values between the block's warps therefore needs a barrier between two items:
shown here from the sources (a lost race would not fail every run)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2509_01827_gb300", "csrc")


def _block(text, at):
    """text between the braces that open at or after `at`."""
    i = text.index("{", at)
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
        if depth == 0:
            return text[i + 1:j - 1]


def _sources():
    out = {}
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        out[os.path.basename(f)] = re.sub(r"//[^\n]*", "", open(f).read())
    return out


def _functions(src):
    """name -> body of the device functions defined in a source."""
    fns = {}
    for m in re.finditer(r"__device__[^;{}()]*?\b(\w+)\s*\([^{};]*?\)\s*\{", src):
        fns[m.group(1)] = _block(src, m.end() - 1)
    return fns


def _shares(name, fns, seen=()):
    """Whether a device function, or one that it calls, shares memory between warps."""
    body = fns.get(name)
    if body is None or name in seen:
        return False
    if "__shared__" in body or "__syncthreads" in body:
        return True
    return any(_shares(c, fns, seen + (name,)) for c in set(re.findall(r"\b(\w+)\s*(?:<[^<>;]*>)?\(", body)))


def _cases():
    src = _sources()
    common = {}
    for f, s in src.items():
        if f.endswith(".cuh"):
            common.update(_functions(s))
    for f, s in src.items():
        for m in re.finditer(r"\b(k_\w+_batch)\(BatchDev b[^)]*\)\s*\{", s):
            yield pytest.param(_block(s, m.end() - 1), {**common, **_functions(s)}, id=m.group(1))


@pytest.mark.parametrize("kernel,fns", list(_cases()))
def test_a_barrier_between_items(kernel, fns):
    loop = _block(kernel, kernel.index("for ("))
    stage = loop.index("stage_member")
    calls = re.findall(r"\b(\w+)\s*(?:<\w+>)?\((?:sd|smem)\b", loop[stage:])
    assert calls, loop
    if any(_shares(c, fns) for c in calls):
        last = max(loop.rindex(c + "(") if c + "(" in loop else loop.rindex(c + "<") for c in calls)
        assert "__syncthreads();" in loop[last:]


def test_loaded_node_list_waits_for_the_ring():
    """The march lists a tile's loaded nodes in the memory of its row ring, at
    positions that other lanes' rows held: votes and shuffles order no memory, so a
    warp barrier stands between the ring's last use and the list's first write."""
    body = _functions(_sources()["step_fp32.cu"])["march32_tile"]
    last_use = max(body.rindex("ring.of("), body.rindex("cp_async_wait<0>"))
    assert "__syncwarp();" in body[last_use:body.index("list[at++]")]
