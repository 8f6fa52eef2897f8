"""Kernels that begin while the launch before them still writes (those that call
pdl_wait) read nothing of it through __ldg, which promises that the memory is
constant for the kernel's whole lifetime: the units that hold such kernels are
searched for it.  The training kernels' samples are the caller's, complete before
the first launch, and may be read so."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_06273_gb300", "csrc")
CALLERS_OWN = {"af_mlp.cu": {"src + j", "reinterpret_cast<const float4 *>(src) + q"}}


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _with_includes(name, seen):
    if name in seen:
        return seen
    seen.add(name)
    for inc in re.findall(r'#include "(af_[a-z0-9_]+\.cuh)"', _code(name)):
        if inc != "af_common.cuh":  # its own loads are those of kernels launched without the attribute
            _with_includes(inc, seen)
    return seen


def _arguments(code, call):
    for m in re.finditer(re.escape(call) + r"\(", code):
        depth, k = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(code[k], 0)
            k += 1
        yield code[m.end():k - 1].strip()


def test_overlapping_kernels_do_not_promise_constant_memory():
    files = set()
    for name in os.listdir(CSRC):
        if name != "af_common.cuh" and re.search(r"\bpdl_wait\(\)", _code(name)):
            _with_includes(name, files)
    assert {"af_flux.cu", "af_pointvalue.cuh", "af_eg2_arc.cuh", "af_mlp.cu"} <= files
    for name in sorted(files):
        loads = set(_arguments(_code(name), "__ldg")) - CALLERS_OWN.get(name, set())
        assert not loads, (name, loads)
        # cell_ubar_global's loads are __ldg's: for kernels launched the ordinary way
        assert not re.search(r"\bcell_ubar_global\(", _code(name)), name
