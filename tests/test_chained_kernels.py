"""Kernels launched with programmatic stream serialization may start while the
launch before them still runs.  Only griddepcontrol.wait makes what earlier
kernels wrote visible, so each of them waits, unconditionally, before it lets
the next one start and before it reads or writes memory (CPU, from the sources)."""
from __future__ import annotations

import glob
import os
import re

from paper_2110_11226_gb300 import build


def _sources():
    out = {}
    for f in sorted(glob.glob(os.path.join(build.CSRC, "*.cu*"))):
        if not f.endswith("gp_fast.cuh"):
            with open(f) as s:
                out[os.path.basename(f)] = re.sub(r"//[^\n]*", "", s.read())
    return out


def _body(text, kernel):
    at = re.search(rf"__global__[^;{{]*?\b{kernel}\s*\(", text)
    if not at:
        return None
    i = text.index("{", at.end())
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
        if depth == 0:
            return text[i + 1:j - 1]


def test_every_chained_kernel_waits_first():
    src = _sources()
    kernels = set()
    for text in src.values():
        for name in re.findall(r"launch_chained\(\s*(\w+)", text):
            # a local name for an instance
            alias = re.search(rf"auto {name} = (\w+)", text)
            kernels.add(alias.group(1) if alias else name)
    kernels.discard("void")  # the launcher's own declaration
    assert {"compile_kernel", "order_kernel", "eval_kernel", "grad_kernel", "finalize_kernel"} <= kernels
    for k in kernels:
        body = next(b for b in (_body(t, k) for t in src.values()) if b is not None)
        # its statements at the top level, blocks left out
        flat, depth = "", 0
        for ch in body:
            depth += {"{": 1, "}": -1}.get(ch, 0)
            flat += ch if depth == 0 and ch != "}" else (";" if ch == "}" and depth == 0 else "")
        statements = [" ".join(s.split()) for s in flat.split(";")]
        assert statements.count("griddep_wait()") == 1, k
        before = statements[:statements.index("griddep_wait()")]
        assert "griddep_launch()" not in before, k
        assert body.count("griddep_wait") == 1 and body.count("griddep_launch") == 1, k
        for s in before:  # declarations and index arithmetic only
            assert not re.search(r"\b(return|for|while|if)\b|atomic|__ldg|\ba\.\w+\s*\[", s), (k, s)
