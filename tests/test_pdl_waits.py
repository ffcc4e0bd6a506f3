"""Programmatic launches, read from the sources: a kernel that is launched so before its
predecessor has ended touches no memory before the wait (or the acquire) that makes what came
before it visible, and the trigger is used nowhere but in the call that releases it."""
import glob
import os
import re

import paper_2403_14244_gb300

CSRC = os.path.join(os.path.dirname(paper_2403_14244_gb300.__file__), "csrc")


def _kernels():
    """(name, statements of the body) of every __global__ function."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s+)?(\w+)\s*\([^{;]*\)\s*\{",
                             text):
            depth, at = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[at], 0)
                at += 1
            yield m.group(1), text[m.end():at - 1]


def test_waits_come_first():
    seen = {}
    for name, body in _kernels():
        if "pdl_" not in body:
            continue
        first = next(s.strip() for s in body.split(";") if not re.match(r"\s*(constexpr|using|static_assert|extern|__shared__)\b", s))
        assert first in ("pdl_wait()", "pdl_behind(started)", "pdl_ahead(started)"), (name, first)
        if "pdl_behind" in body:
            assert body.count("pdl_wait()") >= 1, name  # what follows it in the stream follows both
        seen[first] = seen.get(first, 0) + 1
    assert seen.get("pdl_wait()", 0) > 15 and seen["pdl_behind(started)"] == 1
    text = "".join(open(p).read() for p in glob.glob(os.path.join(CSRC, "*.cu*")))
    assert len(re.findall(r"griddepcontrol\.launch_dependents", text)) == 1
