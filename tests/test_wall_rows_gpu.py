"""The wall blocks of the step kernels and the kernel of odd lattices, where
they can go wrong: lattices that leave lanes, blocks or interior rows empty, and
a Newton solve that FP32 does not settle."""
import numpy as np
import pytest

from gpu_helpers import field_errors, make_pair, set_both
from paper_2304_04214_gb300.inputs import noise

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("inlet", [1, 0])
@pytest.mark.parametrize("precision,tol", [("fp32", 1.5e-5), ("fp16", 1.5e-3), ("bf16", 1.2e-2)])
@pytest.mark.parametrize("shape", [(3, 4, 2), (33, 4, 1), (64, 6, 3), (65, 8, 2), (127, 6, 2), (129, 10, 3)])
def test_ragged_lattices_match_the_oracle(shape, precision, tol, inlet):
    """Two steps (both traversal directions) from a perturbed state: fields, and
    u_tau of every wall cell.  Tolerances: those of the one-step parity tests
    times 1.5 (two steps); u_tau follows the velocity."""
    nx, ny, nz = shape
    o, g = make_pair(nx, ny, nz, n_modes=12, seed=6, precision=precision, inlet=inlet)
    g.step_kernel = "cell"
    set_both(o, g, o.state() * (1.0 + 0.02 * noise((19, nz, ny, nx), seed=8)))
    o.step(2)
    g.step(2)
    g.sync()
    er, eu = field_errors(o, g)
    assert er < tol and eu < tol, (er, eu)
    uo = o.utau().reshape(2, nz, nx)
    assert np.max(np.abs(g.utau() - uo)) < 2 * tol * np.max(uo)


@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16", "fp16row"])
@pytest.mark.parametrize("shape", [(64, 8, 3), (68, 4, 2), (132, 6, 2), (128, 28, 28), (128, 28, 27)])
def test_one_launch_and_side_stream_steps_are_bit_identical(shape, precision):
    """Small lattices (up to 100,000 cells: all but the fourth) run the wall blocks inside
    the step's launch, the staged kernel and larger lattices beside it; x-slabs
    of a channel may fall on either side."""
    nx, ny, nz = shape
    got = []
    for kernel in ("pair", "quad") + (("staged",) if nx % 8 == 0 else ()):
        o, g = make_pair(nx, ny, nz, n_modes=12, seed=6, precision=precision)
        set_both(o, g, o.state() * (1.0 + 0.02 * noise((19, nz, ny, nx), seed=8)))
        g.step_kernel = kernel
        g.step(3)
        got.append((g.populations(), g.utau()))
        g.close()
    for f, u in got[1:]:
        assert np.array_equal(f, got[0][0]) and np.array_equal(u, got[0][1])


@pytest.mark.parametrize("kernel,nx", [("pair", 32), ("cell", 31), ("quad", 32), ("staged", 32)])
def test_newton_from_far_above_the_root(kernel, nx):
    """A channel almost at rest (velocities of 1e-8 .. 1e-7, exact in FP32 as
    differences of populations): u_tau is a thousand times below the initial
    guess, twelve FP32 Newton steps do not reach it and the FP64 solve takes
    over.  One cell per thread: u_hat and u_2 are exact up to the normalization
    of e_x and one division (1e-7 relative), and u_tau ~ sqrt(u_hat) here, so
    1e-5 is ample.  The packed kernels sum u_2 population by population, which
    leaves of so small a velocity only its order: there the solve has to settle,
    within a factor of two."""
    ny, nz = 8, 6
    o, g = make_pair(nx, ny, nz, n_modes=0, inlet=0)
    rng = np.random.Generator(np.random.PCG64(3))
    f = np.empty((19, nz, ny, nx))
    w = np.full(19, 1.0 / 36.0)
    w[9], w[[2, 6, 8, 10, 12, 16]] = 1.0 / 3.0, 1.0 / 18.0
    f[:] = w.astype(np.float32).astype(np.float64)[:, None, None, None]
    ulp = 2.0 ** -28                                     # of an FP32 value near 1/18
    for plus, minus in ((10, 8), (16, 2)):
        n = rng.integers(3, 20, size=(nz, ny, nx))
        f[plus] += n * ulp
        f[minus] -= n * ulp
    o.set_state(f)
    g.set_populations(f)
    g.step_kernel = kernel
    o.step(1)
    g.step(1)
    g.sync()                                             # LBM_ENOTCONV would raise
    uo = o.utau().reshape(2, nz, nx)
    assert np.max(uo) < 1e-5
    if kernel == "cell":
        assert np.allclose(g.utau(), uo, rtol=1e-5, atol=0.0)
    else:
        r = g.utau() / uo
        assert 0.5 < r.min() and r.max() < 2.0


@pytest.mark.parametrize("inlet", [1, 0])
@pytest.mark.parametrize("precision,tol", [("fp16", 1.5e-3), ("bf16", 1.2e-2), ("fp16row", 1.5e-3)])
@pytest.mark.parametrize("shape", [(1026, 8, 14), (898, 10, 12), (126, 30, 28), (130, 30, 28)])
def test_rows_of_pairs_match_the_oracle(shape, precision, tol, inlet):
    """16-bit lattices above 100,000 cells with nx = 4m + 2: the last thread of a row has
    one pair of cells, alone in its warp (1026, 130), at a warp's end (126) or within
    one (898).  Two steps with statistics: fields to the two-step tolerance,
    statistics sums per summed term as in the parity tests."""
    nx, ny, nz = shape
    assert nx % 4 == 2 and nx * ny * nz > 100000
    o, g = make_pair(nx, ny, nz, n_modes=8, seed=6, precision=precision, inlet=inlet, stats=1)
    assert g.step_kernel == "pair"
    set_both(o, g, o.state() * (1.0 + 0.02 * noise((19, nz, ny, nx), seed=8)))
    o.step(2)
    g.step(2)
    g.sync()
    er, eu = field_errors(o, g)
    assert er < tol and eu < tol, (er, eu)
    su = g.stats()[0][..., 0]
    _, uo = o.fields()
    assert np.max(np.abs(su - o.stats()[0].reshape(ny, nx, 7)[..., 0])) < 2 * nz * tol * np.max(np.abs(uo))
