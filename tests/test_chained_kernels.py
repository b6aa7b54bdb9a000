"""Kernels that are brought up while the one before them still runs (chain.cuh) may not read through
the read-only path: what they read is written in their lifetime, and such loads may be moved above the
wait. Checked in the sources: no function that a kernel with chain_begin() reaches uses __ldg or has a
parameter `const T* __restrict__`, and a `__restrict__` parameter of such a kernel is one it only
writes through.
"""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2407_12263_gb300" / "csrc"
OUTPUTS = {"fg_out", "phi", "out", "partials", "result", "fg", "slots", "y"}


def functions(csrc):
    """(file, name, parameters, body) of every function definition under csrc."""
    found = []
    for path in sorted(csrc.glob("*.cu*")):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", path.read_text(), flags=re.S)
        for m in re.finditer(r"\b(\w+)\s*\(((?:[^(){};]|\{\}|\([^(){};]*\))*)\)\s*(?:const\s*)?\{", text):
            if m.group(1) in ("if", "for", "while", "switch", "constexpr", "__launch_bounds__"):
                continue
            depth, i = 1, m.end()
            while depth and i < len(text):
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            found.append((path.name, m.group(1), m.group(2), text[m.end():i]))
    return found


def offences(csrc):
    defs = functions(csrc)
    by_name = {}
    for d in defs:
        by_name.setdefault(d[1], []).append(d)
    kernels = [d for d in defs if re.search(r"\bchain_begin\s*\(\s*\)\s*;", d[3])]
    assert len(kernels) >= 20
    bad, seen, todo = [], set(), list(kernels)
    while todo:
        d = todo.pop()
        if id(d) in seen:
            continue
        seen.add(id(d))
        file, name, params, body = d
        if "__ldg" in body:
            bad.append(f"{file}: {name} uses __ldg")
        for p in params.split(","):
            if "__restrict__" in p and "const" in p.split("__restrict__")[0]:
                bad.append(f"{file}: {name}, parameter{p}")
            elif "__restrict__" in p and d in kernels and p.split()[-1] not in OUTPUTS:
                bad.append(f"{file}: {name} may read through{p}")
        for callee in set(re.findall(r"\b(\w+)\s*(?:<[^;(){}]*>)?\s*\(", body)):
            todo += by_name.get(callee, [])
    reached = {d[1] for d in defs if id(d) in seen}
    return bad, reached


def test_chained_kernels_read_through_ordinary_loads():
    bad, reached = offences(CSRC)
    assert {"step_cell", "pull", "fd_gradient", "trilinear", "restart_cell", "dft_kernel", "conv_tc_kernel"} <= reached
    assert not bad, "\n".join(bad)


@pytest.mark.parametrize("plant", ["const float v = __ldg(q);", None])
def test_the_check_finds_a_read_only_load(tmp_path, plant):
    for path in CSRC.glob("*.cu*"):
        (tmp_path / path.name).write_text(path.read_text())
    glue = tmp_path / "surrogate_glue.cu"
    text = glue.read_text()
    planted = (text.replace("auto lerp = [](", plant + "\n    auto lerp = [](") if plant
               else text.replace("trilinear(const float* q", "trilinear(const float* __restrict__ q"))
    assert planted != text
    glue.write_text(planted)
    assert any("trilinear" in b for b in offences(tmp_path)[0])
