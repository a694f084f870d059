"""Kernels launched with programmatic stream serialisation: no qualified pointer parameters.

Such a kernel may be resident while the kernel before it still writes what it will read after its
dependent-launch wait (griddepcontrol.wait).  A const __restrict__ parameter lets the compiler treat the
array as unchanging for the whole kernel: it may move a load above the wait, or use the non-coherent path,
which has to stay unmodified as long as the kernel lives.
"""
import glob
import os
import re

from paper_2601_16911_gb300 import build as B

WAITS = re.compile(r"\bpdl_wait\s*\(|griddepcontrol\.wait")


def strip_comments(text):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def closing(text, i, pair):
    """Index of the bracket that closes the one at text[i]."""
    depth = 0
    for k in range(i, len(text)):
        depth += (text[k] == pair[0]) - (text[k] == pair[1])
        if depth == 0:
            return k
    raise AssertionError("unbalanced " + pair)


def functions(text):
    """(name, is a kernel, parameters, body) of every device function defined in text."""
    text = re.sub(r"__launch_bounds__\s*\(", "(", strip_comments(text))
    for m in re.finditer(r"\b(__global__|__device__)\b", text):
        brace, semi = text.find("{", m.end()), text.find(";", m.end())
        if brace < 0 or (0 <= semi < brace):
            continue  # a declaration, or a __device__ variable
        head = text[m.end():brace].rstrip()
        if not head.endswith(")"):
            continue
        depth = 0
        for k in range(len(head) - 1, -1, -1):  # the parameter list is the last bracket before the body
            depth += (head[k] == ")") - (head[k] == "(")
            if depth == 0:
                break
        name = re.search(r"(\w+)\s*$", head[:k])
        if name:
            yield name.group(1), m.group(1) == "__global__", head[k:], text[brace:closing(text, brace, "{}") + 1]


def test_kernels_that_wait_for_their_predecessor_take_no_restrict_pointers():
    fns = []
    for f in sorted(glob.glob(os.path.join(B.CSRC, "*.cu")) + glob.glob(os.path.join(B.CSRC, "*.cuh"))):
        with open(f) as h:
            fns += [(os.path.basename(f),) + x for x in functions(h.read())]
    waiting = {name for _, name, _, _, body in fns if WAITS.search(body)}
    while True:  # functions that call one that waits
        more = {name for _, name, _, _, body in fns
                if name not in waiting and any(re.search(r"\b%s\b" % w, body) for w in waiting)}
        if not more:
            break
        waiting |= more
    kernels = [(f, name, par) for f, name, kernel, par, _ in fns if kernel and name in waiting]
    assert {"dg_scalar_stage", "dg_euler_stage", "cg_stage_cells", "cg_node_stage2d", "dg_scalar_steps_tile",
            "mlp_grad_kernel", "mlp_reduce_kernel"} <= {name for _, name, _ in kernels}
    bad = ["%s: %s" % (f, name) for f, name, par in kernels if "__restrict" in par]
    assert not bad, bad
