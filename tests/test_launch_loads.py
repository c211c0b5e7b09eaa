"""Kernels that are set up while the one before still runs: each waits before it
touches memory, and none reads through the read-only path, which is defined only for
data that does not change while the kernel lives."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1706_06989_gb300", "csrc")


def _sources():
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, name)) as f:
                yield name, re.sub(r"//[^\n]*", "", f.read())


def _kernels(text):
    """(name, parameters, body's first statement) of every kernel."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^{;]*?\)\s+)?(\w+)\s*\(", text):
        depth, at = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[at], 0)
            at += 1
        body = text[text.index("{", at) + 1:]
        yield m.group(1), text[m.end():at - 1], body.strip().split(";")[0].strip()


def test_kernels_wait_first_and_load_coherently():
    waiting, launched = set(), set()
    for name, text in _sources():
        launched |= set(re.findall(r"\blaunch\(c, (k_\w+)", text))
        for kernel, params, first in _kernels(text):
            if first != "pdl_wait()":
                assert "pdl_wait" not in first, (name, kernel)
                continue
            waiting.add(kernel)
            for p in params.split(","):
                assert not (p.strip().startswith("const ") and "__restrict__" in p), (name, kernel, p.strip())
        if "pdl_wait" in text:
            assert "__ldg" not in text and "ld.global.nc" not in text, name
    assert launched and launched <= waiting, launched - waiting
    assert len(waiting) > 60
