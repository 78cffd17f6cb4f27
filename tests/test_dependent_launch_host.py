"""Kernels that may start while the one before drains read what kernels write by
coherent loads: a read-only load (__ldg, or a const __restrict__ parameter) promises
data that does not change while the kernel lives."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1204_3425_gb300", "csrc")
TABLES = {"ptr", "npos", "list", "su", "sd", "boff", "bcnt", "ent", "p", "h"}   # written when a handle is made


def _kernels(text):
    """{name: (parameters, body)} of every __global__ function."""
    out = {}
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        params, j = text[m.end():i - 1], text.index("{", i)
        depth, k = 1, j + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[k], 0)
            k += 1
        out[m.group(1)] = (params, text[j:k])
    return out


@pytest.mark.parametrize("src", ["hv_phases.cu", "kernels.cu"])
def test_dependent_kernels_read_vectors_by_coherent_loads(src):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, src)).read())
    kernels = _kernels(text)
    names = {n for n, (_, body) in kernels.items() if "grid_dep_wait()" in body}
    launched = set(re.findall(r"launch_on\(\s*\w+,\s*(\w+)", text))
    assert launched and launched <= names               # every dependent launch waits
    for n in names:
        params, body = kernels[n]
        ro = re.findall(r"const\s+[\w:]+(?:\s+\w+)?\s*\*\s*__restrict__\s+(\w+)", params)
        assert set(ro) <= TABLES, (n, ro)
        for a in re.findall(r"__ldg\(([^()]*(?:\([^()]*\))?)", body):
            assert set(re.findall(r"\b[a-zA-Z_]\w*", a)) & TABLES, (n, a)
        for f in ("__ldcs", "__ldcg"):
            assert f not in body, (n, f)
