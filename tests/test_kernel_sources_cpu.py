"""Launches may overlap the end of the kernel before them, so every kernel has to wait for it before anything else."""
import glob
import os
import re

import paper_2608_02168_gb300

CSRC = os.path.join(os.path.dirname(paper_2608_02168_gb300.__file__), "csrc")


def _skip_parens(s, i):
    depth = 0
    while True:
        depth += {"(": 1, ")": -1}.get(s[i], 0)
        i += 1
        if depth == 0:
            return i


def test_every_kernel_begins_with_pdl_begin():
    kernels = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        s = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__", s):
            i = m.end()
            bounds = re.compile(r"\s*(?:void\s+)?__launch_bounds__\s*").match(s, i)
            if bounds:
                i = _skip_parens(s, bounds.end())
            i = _skip_parens(s, s.index("(", i))
            body = re.compile(r"\s*([{;])\s*(pdl_begin\(\);)?").match(s, i)
            assert body, (path, s[m.start():m.start() + 120])
            if body.group(1) == "{":
                assert body.group(2), (os.path.basename(path), s[m.start():m.start() + 120])
                kernels += 1
    assert kernels > 100
