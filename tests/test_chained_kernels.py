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


def kernel_bodies():
    """name -> the first statements of each __global__ function of that name."""
    out = {}
    for text in sources():
        for m in re.finditer(r"__global__", text):
            head = text[m.end():text.index("{", m.end())]
            head = re.sub(r"__launch_bounds__\s*\((?:[^()]|\([^()]*\))*\)", "", head)
            name = re.search(r"(\w+)\s*\(", head.split("void", 1)[1]).group(1)
            body = text[text.index("{", m.end()) + 1:][:400]
            out.setdefault(name, []).append(body)
    return out


def test_chained_kernels_wait_first():
    bodies = kernel_bodies()
    launched = set()
    for text in sources():
        for m in re.finditer(r"\blaunch_(?:chained|class)\s*\(", text):
            args = text[m.end():m.end() + 200]
            launched |= {k for k in bodies if re.search(r"\b%s\b" % k, args.split(";")[0])}
    assert {"advance_kernel", "plan_kernel", "stats_big_kernel", "warp_tile_kernel"} <= launched
    late = sorted(k for k in launched for b in bodies[k] if b.split(";")[0].strip() != "chain_wait()")
    assert not late, late
