"""What a step launches, counted by the library itself, and lattices on which the
kernels of named and automatic choice differ, against each other."""
import ctypes as ct

import numpy as np
import pytest

from gpu_helpers import make_pair, set_both
from paper_2304_04214_gb300.inputs import noise

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _launches(g, steps):
    """Kernels the handle launches in so many steps (a read starts the count again)."""
    ms, nk, n = ct.c_double(), ct.c_long(), ct.c_long()
    g.lib.lbm_profile_read(g.h, ct.byref(ms), ct.byref(nk), ct.byref(n))
    g.step(steps)
    g.lib.lbm_profile_read(g.h, ct.byref(ms), ct.byref(nk), ct.byref(n))
    return n.value


@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16", "fp16row"])
def test_quad_by_name_runs_beside_the_wall_kernel_on_any_lattice(precision):
    """Small lattices too: QUAD has no wall rows, so a step by that name is two
    launches, where PAIR and AUTO take one."""
    from paper_2304_04214_gb300.channel import LBMChannel
    g = LBMChannel(64, 16, 8, n_modes=0, inlet=False, precision=precision)
    for kernel, want in (("quad", 2), ("pair", 1), ("auto", 1), ("staged", 2), ("cell", 1)):
        g.step_kernel = kernel
        assert _launches(g, 4) == 4 * want, kernel
    g.close()


@pytest.mark.parametrize("precision", ["fp16", "bf16", "fp16row"])
@pytest.mark.parametrize("shape", [(126, 30, 28), (66, 40, 42), (602, 8, 22)])
def test_pair_by_name_gives_the_bits_of_four_cells_a_thread(shape, precision):
    """16-bit lattices of nx = 4m + 2 above 100,000 cells: AUTO takes four cells a
    thread, PAIR two; the last thread of a row at a warp's end, in its middle and
    between."""
    nx, ny, nz = shape
    assert nx * ny * nz > 100000
    got = []
    for kernel in ("auto", "pair"):
        o, g = make_pair(nx, ny, nz, n_modes=8, seed=6, precision=precision, stats=1)
        g.step_kernel = kernel
        set_both(o, g, o.state() * (1.0 + 0.02 * noise((19, nz, ny, nx), seed=8)))
        g.set_sponge(nx // 10, 0.05)
        g.step(3)
        got.append((g.populations(), g.utau(), g.stats()[0]))
        g.close()
    for x, y in zip(*got):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("precision,shape,want", [
    ("fp16", (66, 32, 47), 2), ("fp32", (8, 110, 110), 2), ("fp32", (33, 40, 70), 2), ("bf16", (34, 48, 60), 2),
    ("fp32", (48, 48, 42), 1), ("fp16row", (64, 32, 32), 1), ("fp16", (129, 16, 40), 1)])
def test_lattices_whose_blocks_do_not_fit_at_once_step_in_two_launches(precision, shape, want):
    from paper_2304_04214_gb300.channel import LBMChannel
    g = LBMChannel(*shape, n_modes=0, inlet=False, precision=precision)
    assert _launches(g, 4) == 4 * want
    g.close()


@pytest.mark.parametrize("inlet", [True, False])
@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16", "fp16row"])
@pytest.mark.parametrize("nx,ny,nz", [(65, 16, 8), (129, 6, 11), (64, 16, 8), (66, 8, 15), (33, 12, 9), (301, 4, 7)])
def test_one_launch_and_two_give_the_same_bits(nx, ny, nz, precision, inlet):
    """A state that repeats in z with a period of nz planes (an inlet without modes is
    uniform in z) stays so, plane for plane, in a lattice of many periods: the short
    one steps in one launch, the long one with its wall rows on the side stream.
    Three steps (both traversal directions), with statistics."""
    from paper_2304_04214_gb300.channel import LBMChannel
    reps = 100000 // (nx * ny * nz) + 1
    f = None
    got = []
    for n in (1, reps):
        g = LBMChannel(nx, ny, n * nz, n_modes=0, inlet=inlet, precision=precision, stats_every=1)
        if f is None:
            f = g.populations() * (1.0 + 0.02 * noise((19, nz, ny, nx), seed=8))
        g.set_populations(np.tile(f, (1, n, 1, 1)))
        g.step(3)
        got.append((g.populations(), g.utau()))
        g.close()
    (f1, u1), (f2, u2) = got
    assert np.array_equal(np.tile(f1, (1, reps, 1, 1)), f2)
    assert np.array_equal(np.tile(u1, (1, reps, 1)), u2)


@pytest.mark.parametrize("precision", ["fp16", "bf16", "fp16row"])
@pytest.mark.parametrize("nx,ny,nz", [(3, 6, 9), (15, 4, 5), (21, 8, 11), (31, 16, 10)])
def test_narrow_odd_rows_give_the_same_bits_in_blocks_of_any_width(nx, ny, nz, precision):
    """As above for rows of at most 32 cells: the short lattice in blocks of 64 columns,
    the middle one in one launch of blocks of 32, the long one in two launches."""
    test_one_launch_and_two_give_the_same_bits(nx, ny, nz, precision, True)
    from paper_2304_04214_gb300.channel import LBMChannel
    f = None
    got = []
    for n in (1, 100000 // (32 * ny * nz)):
        g = LBMChannel(nx, ny, n * nz, n_modes=0, precision=precision)
        if f is None:
            f = g.populations() * (1.0 + 0.02 * noise((19, nz, ny, nx), seed=8))
        g.set_populations(np.tile(f, (1, n, 1, 1)))
        g.step(3)
        got.append((g.populations(), g.utau()))
        g.close()
    n = got[1][0].shape[1] // nz
    assert np.array_equal(np.tile(got[0][0], (1, n, 1, 1)), got[1][0])
    assert np.array_equal(np.tile(got[0][1], (1, n, 1)), got[1][1])


def test_wall_rows_alone_are_one_launch():
    """Odd FP32 lattices of ny = 4 above 100,000 cells: no interior kernel, none counted."""
    from paper_2304_04214_gb300.channel import LBMChannel
    g = LBMChannel(1001, 4, 30, n_modes=0, inlet=False)
    assert _launches(g, 4) == 4
    g.close()
