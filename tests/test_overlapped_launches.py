"""A kernel whose start is overlapped with the kernels before it (`launch`) must not read its inputs
as read-only for its lifetime: no __ldg and no `const ... __restrict__` parameter (source check)."""
import glob
import os
import re

from paper_2409_18122_gb300 import build as B


def _sources():
    return {os.path.basename(f): open(f).read() for f in glob.glob(os.path.join(B.CSRC, "*.cu*"))}


def _kernels(text):
    """{name: (parameters, body)} of the kernels defined in a source file."""
    out = {}
    for m in re.finditer(r"__global__ void(?:\s+__launch_bounds__\((?:[^()]|\([^()]*\))*\))?\s+(k_\w+)\(", text):
        end = text.index("{", m.end())
        depth, i = 1, end + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        out[m.group(1)] = (text[m.end():end], text[end:i])
    return out


def test_overlapped_kernels_read_coherently():
    src = _sources()
    overlapped = {n for s in src.values() for n in re.findall(r"\blaunch\((k_\w+)", s)}
    plain = {n for s in src.values() for n in re.findall(r"\blaunch_spread\((k_\w+)", s)}
    kernels = {n: k for s in src.values() for n, k in _kernels(s).items()}
    assert len(overlapped) >= 25 and overlapped <= set(kernels) and not overlapped & plain
    for n in sorted(overlapped):
        params, body = kernels[n]
        assert not re.search(r"const [\w ]+\*\s*__restrict__", params), n
        assert "__ldg" not in body, n


def test_every_kernel_waits_before_anything_else():
    for name, text in _sources().items():
        for n, (_, body) in _kernels(text).items():
            assert re.match(r"\{(\s*//[^\n]*)?\s*pdl_begin\(\);", body), n
