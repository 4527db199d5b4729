"""Kernels launched with chain_launch start before their predecessors on the stream have ended.  Each of them must wait for
them before it ends itself: the end of the last kernel is all that a later call or a reader of the results waits for.  Read
off the sources, so that it runs without a GPU."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_23436_b200", "csrc")


def block(text, at):
    """The braced block that begins at or behind `at`."""
    at = text.index("{", at)
    depth = 0
    for i in range(at, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[at:i + 1]
    raise AssertionError("unbalanced braces")


def kernels_and_chained():
    """(file, kernel) -> body of every kernel, and those that a chain_launch of the same file names."""
    bodies, chained = {}, set()
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        name = os.path.basename(path)
        text = re.sub(r"//[^\n]*", "", open(path).read())
        mine = set()
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^{};]*?\)\s*)?(\w+)\s*\(", text):
            bodies[name, m.group(1)] = block(text, m.end())
            mine.add(m.group(1))
        for m in re.finditer(r"\bchain_launch\(", text):
            start = text.rfind("\ntemplate", 0, m.start()), text.rfind("\nstatic", 0, m.start()), text.rfind("\ncudaError_t", 0, m.start())
            first = text[m.end():text.index("dim3", m.end())] if "dim3" in text[m.end():m.end() + 300] else text[m.end():m.end() + 300]
            if first.lstrip().startswith("kern"):
                first = text[max(start):m.start()]
            named = {k for k in mine if re.search(r"\b%s\b" % k, first)}
            assert named, "%s: which kernel is launched at %r?" % (name, text[m.start():m.start() + 80])
            chained |= {(name, k) for k in named}
    return bodies, chained


BODIES, CHAINED = kernels_and_chained()


def test_the_chained_kernels_are_found():
    assert {k for _, k in CHAINED} >= {"apply_w_kernel", "apply_out_kernel", "sweep_kernel", "cls_row_kernel", "close_kernel", "merge_kernel",
                                       "reverse_kernel", "assemble_kernel", "bwd_w_fix_kernel", "apply_w_f32_kernel", "apply_out_mma_kernel"}


@pytest.mark.parametrize("key", sorted(CHAINED), ids=lambda k: "%s-%s" % k)
def test_a_chained_kernel_waits_for_its_predecessors(key):
    body = BODIES[key]
    assert "chain_wait()" in body
    # on every way out: nothing returns in front of the wait, unless it waits there
    for m in re.finditer(r"\breturn\b", body):
        assert "chain_wait()" in body[:m.start()]
