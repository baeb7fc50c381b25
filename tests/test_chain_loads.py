"""Kernels launched programmatically dependent (launch_chain, csrc/common.cuh) are alive while the
kernels before them still write.  ld.global.nc is defined only for data that nothing writes in
the kernel's whole life, so these kernels may use it (__ldg, const __restrict__) for the plan's constants
alone.  Checked on the sources: no GPU needed."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1504_02897_gb300", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))

# the plan's constants by the names the kernels give them, written before the plan is first used (the node
# scales: by an ordinary launch)
CONSTANT_LOADS = {"a.units", "a.nodes", "a.dest", "red", "src", "ps", "l0", "scale", "g.dcx2", "sy.em1"}
CONSTANT_PARAMS = {
    "columns.cu": {"red", "off", "pos", "scale"},
    "nufft.cu": {"l0", "psi", "scale", "vis"},
    "fft_core.cuh": {"tw"},
}


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _kernels(text):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\((?:[^()]|\([^()]*\))*\))*\)\s*)?(\w+)\s*\(",
                         text):
        def matched(start, opening, closing):
            depth, i = 1, start
            while depth:
                depth += (text[i] == opening) - (text[i] == closing)
                i += 1
            return i
        end = matched(m.end(), "(", ")")
        brace = text.index("{", end)
        yield m.group(1), text[m.end():end - 1], text[brace:matched(brace + 1, "{", "}")]


@pytest.mark.parametrize("name", FILES)
def test_noncoherent_loads_are_of_plan_constants(name):
    # (load_taps' argument `src` holds kernel values: checked where it is called)
    text = _source(name)
    for arg in re.findall(r"__ldg\(([^;]*)", text):
        base = re.match(r"(?:reinterpret_cast<[^>]*>\()?([\w.]+)", arg).group(1)
        assert base in CONSTANT_LOADS, (name, arg)
    for arg in re.findall(r"load_taps<[^>]*>\((\w+)", text):
        assert arg == "ps" or arg.startswith("const"), (name, arg)


@pytest.mark.parametrize("name", FILES)
def test_chain_kernels_mark_only_plan_constants_read_only(name):
    found = 0
    for kernel, params, body in _kernels(_source(name)):
        if "chain_wait()" not in body:
            continue
        found += 1
        for decl in re.findall(r"const\s[^,;=]*?__restrict__\s+(\w+)", params + ";" + body):
            assert decl in CONSTANT_PARAMS.get(name, ()), (name, kernel, decl)
    if name in ("columns.cu", "nufft.cu", "fft_core.cuh", "gpe.cu"):
        assert found >= 2
