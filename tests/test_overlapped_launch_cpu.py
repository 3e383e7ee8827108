"""Kernels whose launch overlaps the end of the kernel before (griddepcontrol.wait) run while
their arguments are still being written.  A __restrict__ pointer argument promises that nobody
else writes its memory for as long as the kernel runs, and allows the compiler to load through it
before the wait or by the non-coherent path; so such a kernel has none.  Read from the sources."""
import os
import re

from paper_1202_6351_gb300 import build as B


def kernels(text):
    """(name, argument list, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\b", text):
        i = m.end()
        name = None
        while True:  # name(args), past __launch_bounds__(...)
            m2 = re.compile(r"(\w+)\s*\(").search(text, i)
            depth, j = 1, m2.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[j], 0)
                j += 1
            if m2.group(1) != "__launch_bounds__":
                name, args = m2.group(1), text[m2.end():j - 1]
                break
            i = j
        k = text.index("{", j)
        depth, e = 1, k + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[e], 0)
            e += 1
        yield name, args, text[k:e]


def test_overlapped_kernels_have_no_restrict_arguments():
    waiting = {}
    for f in sorted(os.listdir(B.CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(B.CSRC, f)).read())
        for name, args, body in kernels(text):
            if "pdl_wait()" in body:
                waiting[name] = args
    assert {"step_kernel", "multi_kernel", "adj_step_kernel", "resident_kernel", "step3_kernel"} <= set(waiting)
    assert [n for n, args in waiting.items() if "__restrict__" in args] == []
