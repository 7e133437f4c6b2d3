"""Source check (no GPU): what an earlier launch wrote is never read as if it were constant.

Kernels of one call may start while the one before still runs.  CUDA allows the non-coherent path (``ld.global.nc``,
``__ldg``, and what the compiler makes of ``const T *__restrict__`` kernel parameters) only for data that nobody writes
while the reading kernel lives, so it is left to the caller's tensors, and there to kernels that cannot be a call's first."""
import glob
import os
import re

from conftest import ROOT

SOURCES = sorted(glob.glob(os.path.join(ROOT, "paper_2502_11494_b200", "csrc", "*.cu*")))
CALLERS = {"keys", "hidden", "pos_in"}
MAY_BE_FIRST = {"pivots_given_kernel"}  # launched behind whatever the caller's stream runs


def _code(path):
    text = open(path).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _kernels(code):
    """(name, parameter list) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", code):
        depth, at = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(code[at], 0)
            at += 1
        yield m.group(1), code[m.end():at - 1]


def test_explicit_non_coherent_loads_are_in_one_place():
    code = {os.path.basename(p): _code(p) for p in SOURCES}
    assert not any("__ldg" in c for c in code.values())
    assert {n: c.count("ld.global.nc") for n, c in code.items() if "ld.global.nc" in c} == {"dart_common.cuh": 1}   # ld_stream
    # by whom: kernels that read the caller's rows behind another launch of the same call, or are launched behind everything
    users = {name for c in code.values() for name in re.findall(r"\n(\w+)\([^{;]*\)\s*\{(?:(?!\n\}).)*ld_stream", c, flags=re.S)}
    assert users == {"score_kernel", "sim_alu_kernel", "gather_varlen_kernel", "gather_kernel"}
    assert "ld_stream<kFirst>" in code["dart_staged.cuh"] and not re.search(r"launch_next\(\s*score_kernel", code["dart_api.cu"])
    entry = code["dart_api.cu"].split("int dart_gather_rows(")[1].split("\n}")[0]
    assert "gather_kernel<true>" in entry


def test_constant_kernel_parameters_are_the_callers_tensors():
    seen = set()
    for path in SOURCES:
        for name, params in _kernels(_code(path)):
            seen.add(name)
            const = set(re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", params))
            assert const <= (set() if name in MAY_BE_FIRST else CALLERS), (name, const)
    assert {"score_kernel", "pivots_given_kernel", "retain_kernel", "gather_kernel", "rank_kernel", "onepass_kernel", "flow_kernel"} <= seen
