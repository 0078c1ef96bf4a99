"""Kernels that may start while the kernel before them in the stream still runs: what they read through the
read-only path, or through a pointer that promises constant memory, has to be constant for as long as they
run, which is not so for what their predecessors write.  Read from the sources: no GPU needed."""
import glob
import os
import re

from paper_2101_06983_b200 import _build


def _kernels():
    for path in sorted(glob.glob(os.path.join(_build.CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        starts = [m.start() for m in re.finditer(r"\b__global__\b", text)]
        for a, b in zip(starts, starts[1:] + [len(text)]):
            body = text[a:b]
            m = re.search(r"\b(\w+_kernel)\s*\(", body)
            if m and body.find("{") >= 0:
                yield os.path.basename(path), m.group(1), body


def test_kernels_that_start_early_read_nothing_as_constant():
    early = [(f, n, b) for f, n, b in _kernels() if re.search(r"\bdep_wait\(\)", b)]
    names = {n for _, n, _ in early}
    assert {"strip_logit_kernel", "strip_row_kernel", "strip_grad_kernel", "apply_kernel", "small_kernel",
            "lse_combine_kernel", "row_dot_kernel", "cosine_bwd_kernel"} <= names
    for f, n, body in early:
        signature = body[:body.index("{")]
        assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", signature), (f, n)
        assert "__ldg(" not in body, (f, n)


def test_kernels_wait_before_they_are_left():
    """A kernel that lets its successor start early waits for its own predecessor: its completion then stands
    for that of everything before it."""
    for f, n, body in _kernels():
        if "dep_release()" in body and n != "pos_anchor_kernel":      # launched without the attribute
            assert "dep_wait()" in body, (f, n)
