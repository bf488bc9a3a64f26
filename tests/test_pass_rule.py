"""Lanes and row bands of a staged-cell pass (host rule): a batch's do not depend on the order of its
cameras, a view's alone are those of any number of equal ones, and the closest rays of a batch decide."""
import ctypes
import itertools
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = """
#include "vr_pass.h"
extern "C" void shape(const double* spacing, int n, int f32, int* out) {
    const double c[3] = {32, 32, 32};
    std::vector<vr::CamDev> cams((size_t)n);
    for (int i = 0; i < n; ++i) {  // orthographic, the pixels `spacing` voxels apart
        vr::CamDev d{};
        d.right[0] = d.up[1] = d.fwd[2] = 1.0;
        d.du = d.dv = spacing[i];
        cams[(size_t)i] = d;
    }
    const vr::PassShape p = vr::pass_rule(c, cams.data(), n, f32 != 0);
    out[0] = p.group;
    out[1] = p.bands;
}
"""


@pytest.fixture(scope="module")
def shape(tmp_path_factory):
    from paper_1012_2909_gb300 import _build
    d = tmp_path_factory.mktemp("pass")
    (d / "t.cpp").write_text(SOURCE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    subprocess.run([shutil.which("g++") or "c++", "-std=c++17", "-shared", "-fPIC", "-I", _build.INCLUDE, "-I",
                    _build.CSRC, "-I", cuda, str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    lib = ctypes.CDLL(str(d / "t.so"))

    def call(spacing, f32):
        out = (ctypes.c_int * 2)()
        lib.shape((ctypes.c_double * len(spacing))(*spacing), len(spacing), int(f32), out)
        return tuple(out)

    return call


@pytest.mark.parametrize("f32,limit", [(True, 3.0), (False, 1.0)])
def test_shape(shape, f32, limit):
    assert shape([limit], f32)[0] == 4 and shape([limit * 1.001], f32)[0] == 8
    assert shape([0.01], f32)[1] == 64 and shape([10.0], f32)[1] == 1
    for s in (0.1, 0.4, 0.9, 1.5, 2.9, 8.0):
        assert shape([s], f32) == shape([s] * 25, f32)
    mixed = (0.2, 5.0, 20.0)
    assert len({shape(list(p), f32) for p in itertools.permutations(mixed)}) == 1
    assert shape([0.2, 20.0], f32)[0] == 4 and shape([4.0, 20.0], f32)[0] == 8
