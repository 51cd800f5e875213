"""Kernels that may be set up while their predecessor runs (launch_chained) wait for it, in every
thread and before anything else: a grid whose predecessor lets it start early has no other order
with what ran before."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1006_0532_gb300", "csrc")


def sources():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh", ".h")):
            text = open(os.path.join(CSRC, name)).read()
            yield re.sub(r"//[^\n]*", "", text)


def without_bounds(head):
    """A kernel's head without __launch_bounds__(...)."""
    at = head.find("__launch_bounds__")
    if at < 0:
        return head
    end, depth = head.index("(", at), 0
    while True:
        depth += {"(": 1, ")": -1}.get(head[end], 0)
        end += 1
        if depth == 0:
            return head[:at] + head[end:]


def kernel_bodies():
    """name -> the first statements of each __global__ function of that name."""
    out = {}
    for text in sources():
        for m in re.finditer(r"__global__", text):
            head = without_bounds(text[m.end():text.index("{", m.end())])
            name = re.search(r"(\w+)\s*\(", head.split("void", 1)[1]).group(1)
            body = text[text.index("{", m.end()) + 1:][:400]
            out.setdefault(name, []).append(body)
    return out


def test_chained_kernels_wait_first():
    bodies = kernel_bodies()
    launched = set()
    for text in sources():
        for m in re.finditer(r"\blaunch_chained\s*\(", text):
            args = text[m.end():m.end() + 200]
            launched |= {k for k in bodies if re.search(r"\b%s\b" % k, args.split(";")[0])}
    assert {"advance_kernel", "plan_kernel", "stats_big_kernel", "small_grid_kernel"} <= launched
    late = sorted(k for k in launched for b in bodies[k] if b.split(";")[0].strip() != "chain_wait()")
    assert not late, late
