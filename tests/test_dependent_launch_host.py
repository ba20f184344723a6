"""Kernels launched while their predecessor drains (launch_kernel): each waits for it
before anything else and reads what it may have written with plain loads.  Read
from the sources: a missing wait or a non-coherent load shows as a wrong value
only where the timing allows it."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_13215_gb300", "csrc")


def _code(name):
    src = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)


SOURCES = {n: _code(n) for n in sorted(os.listdir(CSRC)) if n.endswith((".cu", ".cuh"))}
LAUNCHED = sorted({m for s in SOURCES.values() for m in re.findall(r"\blaunch_kernel\((k_\w+)", s)})


def _kernel(name):
    """(parameters, body) of the kernel's definition."""
    for src in SOURCES.values():
        m = re.search(r"__global__\s+void\s+__launch_bounds__\(.*?\)\s*%s\((?P<args>[^{;]*)\)\s*\{" % name, src, re.S)
        if m:
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[i], 0)
                i += 1
            return m.group("args"), src[m.end():i - 1]
    raise AssertionError("no definition of %s" % name)


def test_the_main_path_is_launched_so():
    assert {"k_slice_project", "k_cell_count", "k_tile_write", "k_composite_fwd", "k_composite_bwd", "k_loss_sum",
            "k_adjoint", "k_adam"} <= set(LAUNCHED)


@pytest.mark.parametrize("name", LAUNCHED)
def test_waits_first_and_loads_plainly(name):
    args, body = _kernel(name)
    assert "__restrict__" not in args
    assert "__ldg" not in body and "ld.global.nc" not in body
    before, wait, _ = body.partition("wait_for_previous_kernel();")
    assert wait
    # only declarations and constants ahead of the wait: no load, no early return
    for line in filter(None, (x.strip() for x in before.split(";"))):
        assert re.match(r"(extern )?__shared__|(const|constexpr|static_assert)\b", line), line
        assert "->" not in line and "[" not in line.split("=", 1)[-1] or "__shared__" in line, line


def test_non_coherent_loads_only_where_a_call_allows_them():
    """__ldg only in load_global; its non-coherent form only in the projection, whose call clears the status word
    first, and in the conversion, which is launched plainly."""
    for name, src in SOURCES.items():
        assert len(re.findall(r"__ldg\(|ld\.global\.nc", src)) == (1 if name == "splat_internal.cuh" else 0), name
        assert not re.search(r"const\s+[\w ]+\*\s*__restrict__", src), name
    assert not re.search(r"\blaunch_kernel\(", SOURCES["convert.cu"])
    true = {n: len(re.findall(r"<DT, true>|ld<true>", s)) for n, s in SOURCES.items()}
    assert [n for n, c in true.items() if c] == ["convert.cu", "project.cu"]
    args, body = _kernel("k_slice_project")
    assert "load_geo<DT, true>" in body
    args, body = _kernel("k_adjoint")
    assert "true>" not in body
    call = SOURCES["api.cu"].partition("splat_status splat_slice_project(")[2]
    assert call.index("cudaMemsetAsync(status") < call.index("launch_slice_project(")
