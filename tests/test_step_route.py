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
    (d / "r.cpp").write_text('#include "lbm_route.h"\nextern "C" void route(int kind, int obj, int precision, int nx, '
                             'int ny, int nz, int sms, lbmk::StepRoute *r) '
                             '{ *r = lbmk::step_route(kind, obj, precision, nx, ny, nz, sms); }\n')
    so = str(d / "r.so")
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, "-I", build.INCLUDE,
                    str(d / "r.cpp"), "-o", so], check=True)
    lib = ct.CDLL(so)

    def f(kind, elem, shape, obj=False, precision=None, sms=152):
        r = Route()
        if precision is None:
            precision = _abi.LBM_FP32 if elem == 4 else _abi.LBM_FP16_DEV
        lib.route(kind, int(obj), precision, *shape, sms, ct.byref(r))
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


@pytest.mark.parametrize("elem,shape,one", [
    (4, (64, 32, 32), True), (2, (64, 32, 32), True), (2, (48, 48, 42), True), (4, (130, 24, 32), True),
    (2, (128, 32, 24), True), (4, (63, 32, 32), True),
    # more blocks than the device holds at once
    (2, (66, 32, 47), False), (4, (8, 110, 110), False), (4, (20, 50, 98), False), (2, (34, 48, 60), False),
    (2, (72, 40, 34), False), (4, (33, 40, 70), False), (4, (97, 32, 32), False), (2, (65, 32, 47), False),
    # wall rows only; QUAD's lattices of narrow rows; above the cell count
    (4, (999, 4, 24), True), (2, (16, 60, 100), True), (4, (128, 32, 32), False), (2, (96, 32, 48), False)])
def test_one_launch_where_its_blocks_are_resident(route, elem, shape, one):
    assert bool(route(AUTO, elem, shape).one) == one


def test_one_launch_follows_the_size_of_the_device(route):
    """The same lattice on fewer SMs; and never more blocks than fit, but for wall
    rows alone and QUAD's narrow lattices."""
    assert route(AUTO, 4, (64, 32, 32), sms=64).one and not route(AUTO, 4, (64, 32, 32), sms=63).one
    for nx in range(2, 200):
        for ny, nz in ((6, 60), (16, 40), (40, 40), (90, 90)):
            for elem in (2, 4):
                r = route(AUTO, elem, (nx, ny, nz))
                if r.one and not (elem == 2 and nx % 4 == 0 and nx <= 64):
                    assert r.bx * r.nbx * ny * nz <= 152 * 512


FP16, BF16, ROW = _abi.LBM_FP16_DEV, _abi.LBM_BF16_DEV, _abi.LBM_FP16_ROW


@pytest.mark.parametrize("shape,precision,even", [
    ((602, 60, 48), BF16, True), ((602, 60, 48), ROW, True), ((66, 60, 60), BF16, True), ((126, 30, 28), ROW, True),
    ((222, 60, 60), ROW, True),
    # plain FP16, and rows that warps of 128 columns leave emptier than blocks of 64 or 128
    ((602, 60, 48), FP16, False), ((34, 60, 60), BF16, False), ((18, 100, 100), ROW, False),
    ((130, 48, 48), BF16, False), ((386, 96, 96), ROW, False), ((1026, 8, 14), BF16, False)])
def test_four_cells_a_thread_on_rows_of_pairs(route, shape, precision, even):
    r = route(AUTO, 2, shape, precision=precision)
    assert bool(r.even) == even and r.kind == (QUAD if even else PAIR) and not r.one
    assert not even or r.nbx * 128 <= -(-shape[0] // 64) * 64


@pytest.mark.parametrize("shape,bx,one", [
    ((21, 16, 30), 32, True), ((31, 40, 40), 32, True),      # resident in blocks of 64 columns
    ((21, 48, 90), 16, True), ((29, 58, 58), 16, True),
    ((21, 100, 100), 16, False), ((33, 100, 100), 32, False), ((27, 4, 1000), 16, False)])
def test_narrow_odd_rows_of_16_bit_lattices(route, shape, bx, one):
    r = route(AUTO, 2, shape)
    assert r.split and r.bx == bx and bool(r.one) == one
