"""Which kernels run a step (csrc/lbm_route.h), on the host: the rule is plain
C++, compiled here by itself."""
import ctypes as ct
import os
import shutil
import subprocess

import pytest

from paper_2304_04214_gb300 import _abi, build

CELL, PAIR, QUAD, STAGED, AUTO = (_abi.LBM_KERNEL_CELL, _abi.LBM_KERNEL_PAIR, _abi.LBM_KERNEL_QUAD,
                                  _abi.LBM_KERNEL_STAGED, _abi.LBM_KERNEL_AUTO)


class Route(ct.Structure):
    _fields_ = [("kind", ct.c_int), ("one", ct.c_bool), ("split", ct.c_bool), ("even", ct.c_bool),
                ("bx", ct.c_int), ("nbx", ct.c_int)]


@pytest.fixture(scope="module")
def route(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("route")
    (d / "r.cpp").write_text('#include "lbm_route.h"\nextern "C" void route(int kind, int obj, int elem, int nx, int ny, '
                             'int nz, lbmk::StepRoute *r) { *r = lbmk::step_route(kind, obj, elem, nx, ny, nz); }\n')
    so = str(d / "r.so")
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, "-I", build.INCLUDE,
                    str(d / "r.cpp"), "-o", so], check=True)
    lib = ct.CDLL(so)

    def f(kind, elem, shape, obj=False):
        r = Route()
        lib.route(kind, int(obj), elem, *shape, ct.byref(r))
        return r
    return f


SHAPES = [(64, 32, 32), (64, 4, 1), (70, 16, 6), (136, 12, 5), (1026, 8, 14), (602, 60, 48), (384, 96, 96),
          (66, 60, 60), (18, 100, 100)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("elem", [2, 4])
def test_a_kind_chosen_by_name_runs_as_that_kernel(route, shape, elem):
    for kind in (CELL, PAIR, STAGED) + ((QUAD,) if shape[0] % 4 == 0 else ()):
        r = route(kind, elem, shape)
        assert r.kind == kind and not r.even
        assert not (r.one and kind in (QUAD, STAGED))       # kernels of interior rows only


@pytest.mark.parametrize("shape", SHAPES + [(65, 16, 8), (241, 62, 75), (3, 4, 2)])
@pytest.mark.parametrize("elem", [2, 4])
def test_blocks_cover_the_row_once(route, shape, elem):
    """Every kind: the blocks' columns reach the row's end, the last block holds
    some of it, and a block has at most as many threads as the kernels are built for."""
    nx = shape[0]
    kinds = [AUTO, CELL] + ([PAIR] if nx % 2 == 0 else []) + ([QUAD] if nx % 4 == 0 else [])
    for kind in kinds:
        for obj in (False, True) if elem == 4 else (False,):
            r = route(kind, elem, shape, obj)
            per = {QUAD: 4, PAIR: 2, CELL: 2 if elem == 2 else 1}[r.kind] * r.bx
            assert r.nbx * per >= nx > (r.nbx - 1) * per
            assert r.bx * 2 <= (64 if r.kind == QUAD else 128)
            assert r.split == (r.kind == CELL and elem == 2)
            assert not obj or r.kind in (CELL, PAIR)
            assert nx % 2 == 0 or r.kind == CELL
            assert r.kind != QUAD or nx % 4 == 0 or (r.even and elem == 2)
