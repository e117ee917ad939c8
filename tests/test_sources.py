"""Properties of the CUDA sources that no run can show, read from their text."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_08820_gb300", "csrc")


def _kernels(path):
    """(parameter list, body) of every __global__ function of a file, comments removed."""
    with open(path, encoding="utf-8") as fh:
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", fh.read(), flags=re.S)
    for m in re.finditer(r"\b__global__\b", src):
        start = src.index("{", m.end())
        depth, end = 0, start
        while True:
            depth += {"{": 1, "}": -1}.get(src[end], 0)
            end += 1
            if depth == 0:
                break
        yield src[m.end():start], src[start:end]


def test_overlapping_kernels_read_their_predecessors_data_by_coherent_loads():
    """A kernel launched before its predecessor has ended (it waits with grid_dependency_wait) must not read what
    that one writes through the read-only path: data read so has to stay unchanged for the kernel's whole lifetime. So it
    neither loads by __ldg after the wait nor takes const __restrict__ pointers, from which the compiler may infer such
    loads. (tile_rep is written when a batch is laid out, before any of its steps.)"""
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for params, body in _kernels(path):
            if "grid_dependency_wait" not in body:
                continue
            seen += 1
            where = (os.path.basename(path), params.strip()[-60:])
            frozen = set(re.findall(r"const\s[^,()]*\*\s*__restrict__\s+(\w+)", params)) - {"tile_rep"}
            assert not frozen, where + (frozen,)
            waited = body[body.index("grid_dependency_wait"):]
            assert "__ldg" not in waited and "ld.global.nc" not in waited, where
            assert not re.search(r"const\s[^;=]*\*\s*__restrict__", waited), where
    assert seen >= 15


@pytest.mark.parametrize("read,ok", [("x = src[i];", True), ("x = __ldg(src + i);", False)])
def test_the_scan_sees_what_it_looks_for(tmp_path, read, ok):
    f = tmp_path / "k.cu"
    f.write_text("template <int N>\n__global__ void __launch_bounds__(64) k(const float* src) { // {\n"
                 "  if (N) { grid_dependency_wait(); }\n  " + read + "\n}\nint other() { return 1; }\n")
    (params, body), = _kernels(str(f))
    assert "src" in params and body.endswith("}") and ("__ldg" in body) is not ok and "other" not in body
