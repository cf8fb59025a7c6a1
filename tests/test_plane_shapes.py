"""Launch shapes of the plane pipeline, checked on the host: what its CTAs
take of an SM (shared memory, threads, tensor memory), and that every unit of
the group split has its place.  A host program evaluates the compile-time
constants; no kernel is compiled or launched.
"""

import json
import os
import shutil
import subprocess

import pytest

from tests.test_launch_shapes import CSRC, ROOT, SMEM_PER_CTA, SMEM_PER_SM, _registry


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    lines = ['#include <cstdio>', '#include "exx_ops.cuh"', "using namespace exx;",
             "template <typename T> void show(const char* bc, int n, const char* prec) {",
             "  using K = typename T::PC; using X = typename T::XC;",
             '  std::printf("{\\"bc\\": \\"%s\\", \\"n\\": %d, \\"prec\\": \\"%s\\", \\"ok\\": %d, \\"ry\\": %d, '
             '\\"nt\\": %d, \\"c\\": %d, \\"ng\\": %d, \\"smem\\": %zu, \\"tcols\\": %d, \\"g\\": %d, \\"rows\\": %d, '
             '\\"per_z\\": %d, \\"x_nt\\": %d, \\"x_c\\": %d, \\"x_smem\\": %zu, \\"zb\\": %d, \\"x1\\": %d}\\n", bc, n, '
             'prec, (int)T::plane_ok, T::RY, K::NT, K::MINB, K::NG, K::smem, K::tcols, T::G, K::ROWS, '
             '(int)K::Z::PER, X::NT, X::MINB, X::smem_f, X::ZB, X::X1);',
             "}", "int main() {"]
    for bc, n, args in _registry():
        for prec, R in (("fp32", "float"), ("fp64", "double")):
            lines.append(f'  show<OpsImpl<{R}, {args}>>("{bc}", {n}, "{prec}");')
    lines += ["  return 0;", "}"]
    d = tmp_path_factory.mktemp("plane_shapes")
    src, exe = d / "shapes.cu", d / "shapes"
    src.write_text("\n".join(lines) + "\n")
    subprocess.run([nvcc, "-std=c++17", "-O0", f"-I{CSRC}", f"-I{os.path.join(ROOT, 'include')}",
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [s for s in map(json.loads, out.splitlines()) if s["ok"]]


def test_plane_pipeline_covers_the_grids_it_fits(shapes):
    have = {(s["bc"], s["n"], s["prec"]) for s in shapes}
    assert {("free", n, "fp32") for n in (16, 28, 56, 96, 112, 128, 160)} <= have
    assert {("free", 112, "fp64"), ("periodic", 128, "fp32"), ("slab", 96, "fp64"), ("wire", 96, "fp64")} <= have
    assert not {("free", 160, "fp64"), ("periodic", 192, "fp32"), ("free", 14, "fp32")} & have


def test_plane_ctas_fit_an_sm(shapes):
    for s in shapes:
        smem = s["smem"] + 8 * s["nt"] + 16  # with the static energy partials
        assert smem <= SMEM_PER_CTA and s["nt"] <= 1024 and s["nt"] * s["c"] <= 2048, s
        assert s["c"] == 1 or s["c"] * (smem + 1024) <= SMEM_PER_SM, s
        assert s["per_z"] or s["c"] * s["tcols"] <= 512, s
        assert s["g"] % s["ng"] == 0 and s["rows"] % s["ng"] == 0 and s["nt"] % (32 * s["ng"]) == 0, s
        assert s["ng"] <= 15, s  # named barriers 1..ng


def test_line_kernel_ctas_fit_an_sm(shapes):
    for s in shapes:
        assert s["x_nt"] * s["x_c"] <= 2048 and s["x_smem"] <= 48 * 1024 * 2, s
        assert s["g"] % s["zb"] == 0 and s["x1"] % 2 == 0, s
