"""Kernels that are placed before the one before them has ended (launch_early,
csrc/common.cuh): each waits in its first statement, and none reads by
non-coherent loads, which want memory that nothing writes while the kernel
lives. By reading the sources."""
import os
import re

import paper_1405_7958_gb300.build as build

SOURCES = {os.path.basename(p): open(p).read() for p in build.sources()}
COMMON = open(os.path.join(build.CSRC, "common.cuh")).read()


def kernels(text):
    """name -> body of every kernel of a source file"""
    found = {}
    for part in text.split("__global__")[1:]:
        name = re.match(r"\s*void\s+(?:__launch_bounds__\([^()]*\)\s+)?(\w+)\(", part).group(1)
        start = part.index("\n{", 0) + 2
        found[name] = part[start:part.index("\n}\n", start)]
    return found


def test_early_kernels_wait_first_and_load_coherently():
    early = 0
    for file, text in SOURCES.items():
        bodies = kernels(text)
        for name, body in bodies.items():
            if "start_early()" not in body:
                continue
            early += 1
            assert body.strip().startswith("start_early();"), (file, name)
            for line in body.splitlines():
                assert "__ldg(" not in line or "kGroupTable" in line, (file, name, line)
        for name in re.findall(r"launch_early\((\w+_kernel)\b", text):
            assert "start_early()" in bodies[name], (file, name)
        if "start_early()" in text:
            assert "__restrict__" not in text, file
    assert early >= 25
    assert "__ldg(p" not in COMMON and "__ldg(q" not in COMMON and "__ldg(reinterpret" not in COMMON
