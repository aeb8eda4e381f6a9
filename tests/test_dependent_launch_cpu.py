"""Kernels that start behind a running kernel (launch_behind) live while the
kernels before them still write.  What such a kernel reads it loads plainly: a
load through __ldg or through a const __restrict__ pointer may take the
read-only path or be moved above the wait, which is right only for data that
stays unwritten for the kernel's whole life."""
import os
import re

from paper_2007_00558_gb300 import build

# view descriptors and frame tables, complete before the splat starts, behind
# which the resolve and the crack pass run; the encoder's table, which the host wrote
UNWRITTEN = {"views", "frames", "lut"}


def _functions(path):
    """(signature, body) of every device function and kernel of a source file."""
    s = re.sub(r"//[^\n]*", "", open(path).read())
    for m in re.finditer(r"__(?:global|device)__[^;{}=]*\{", s):
        depth, j = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(s[j], 0)
            j += 1
        yield m.group(0), s[m.end():j]


def test_kernels_behind_a_running_one_load_plainly():
    seen = 0
    for path in build.sources():
        for sig, body in _functions(path):
            if not re.search(r"\b(behind|wait_primary)\(\);", body):
                continue
            seen += 1
            where = os.path.basename(path) + ": " + " ".join(sig.split())
            names = set(re.findall(r"__restrict__\s+(\w+)", sig))
            assert names <= UNWRITTEN, where
            for arg in re.findall(r"__ldg\((\w+)", body):
                assert arg in UNWRITTEN, where
    assert seen >= 15
