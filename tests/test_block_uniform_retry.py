"""A kernel whose threads work together (barriers, shared memory, shuffles) asks once for the whole block
whether its pass is to be rerun: the status can change between two warps' reads, and warps that go on
without the others use shared counts and places that were never set, as indices among other things."""
from __future__ import annotations

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_03707_gb300", "csrc")
TOGETHER = re.compile(r"__syncthreads|__syncwarp|__shared__|_sync\(|\bsync\(\)")


def _functions(text):
    """(name, is a kernel, body) of the functions defined in a source file."""
    text = re.sub(r"//[^\n]*", "", text)
    text = re.sub(r"__launch_bounds__\((?:[^()]|\([^()]*\))*\)", "", text)
    for m in re.finditer(r"(__global__|__device__)[^;{}]*?(\w+)\(([^;{}]*)\)\s*(?:const\s*)?\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        head = text[max(0, m.start() - 40):m.end()]
        yield m.group(2), "__global__" in head, text[m.end():i - 1]


def test_blocks_ask_as_one():
    kernels, askers = {}, {"pass_retrying"}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for name, kernel, body in _functions(open(path).read()):
            if kernel:
                kernels[name] = body
            elif name != "block_retrying" and re.search(r"\bpass_retrying\(", body):
                askers.add(name)
    for name in ("dp_init", "dp_wave", "dp_rows", "rows_thread", "rows_group", "rows_warp", "rows_block", "reach_push", "trace_kernel",
                 "gather_rows"):
        assert name in kernels and TOGETHER.search(kernels[name])
    wrong = [name for name, body in kernels.items()
             if TOGETHER.search(body) and any(re.search(rf"\b{a}\(", body) for a in askers)]
    assert not wrong
