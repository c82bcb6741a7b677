"""What the CUDA sources promise about programmatic launches, read from the text (no GPU).

A kernel that executes ``griddepcontrol.wait`` is ordered after the kernels before it
only through that wait, and what follows it on the stream waits for it alone.  A thread
that returns before the wait takes its block out of that order.
"""
import glob
import os
import re


ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_2606_29563_gb300", "csrc", "*.cu")))


def kernels():
    """(name, body) of every __global__ function, comments left out."""
    for path in SOURCES:
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        for m in re.finditer(r"__global__([^{;]*)\{", text):
            name = [n for n in re.findall(r"(\w+)\s*\(", m.group(1)) if n != "__launch_bounds__"][0]
            at = m.end() - 1
            depth, end = 0, at
            while True:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
                if depth == 0:
                    break
            yield name, text[at:end]


def test_no_kernel_returns_before_its_wait():
    waiting = [(name, body) for name, body in kernels() if "griddepcontrol.wait" in body]
    assert len(waiting) >= 10
    early = [name for name, body in waiting if re.search(r"\breturn\s*;", body[:body.index("griddepcontrol.wait")])]
    assert not early
