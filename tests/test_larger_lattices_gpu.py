"""The kernels and stream orders of lattices above 100,000 cells, whose steps keep the
wall rows on a side stream beside the interior kernel: every kernel against the oracle
and against each other, CUDA graphs, coupling loops, adjoint windows and guard bands on
sizes that leave lanes of a warp, blocks or interior rows empty."""
import ctypes as ct

import numpy as np
import pytest

import test_guard_gpu
from gpu_helpers import field_errors, make_pair, set_both
from paper_2304_04214_gb300.inputs import noise, stg_uniforms

pytestmark = pytest.mark.gpu

# one-step tolerances of the parity tests, for two steps
TOL = {"fp32": 1.5e-5, "fp16": 1.5e-3, "bf16": 1.2e-2, "fp16row": 1.5e-3}
PRECISIONS = list(TOL)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _dp(a):
    return a.ctypes.data_as(ct.POINTER(ct.c_double))


def _perturbed(shape, precision, kernel, inlet=1, sponge=(0, 0.0)):
    nx, ny, nz = shape
    assert nx * ny * nz > 100000
    o, g = make_pair(nx, ny, nz, n_modes=8, seed=6, precision=precision, inlet=inlet, stats=1, sponge=sponge)
    g.step_kernel = kernel
    set_both(o, g, o.state() * (1.0 + 0.02 * noise((19, nz, ny, nx), seed=8)))
    return o, g


def _against_the_oracle(shape, precision, kernel, inlet, sponge):
    """Two steps (both traversal directions): fields, u_tau, statistics per summed term."""
    nx, ny, nz = shape
    tol = TOL[precision]
    o, g = _perturbed(shape, precision, kernel, inlet, sponge)
    o.step(2)
    g.step(2)
    g.sync()
    er, eu = field_errors(o, g)
    assert er < tol and eu < tol, (er, eu)
    uo = o.utau().reshape(2, nz, nx)
    assert np.max(np.abs(g.utau() - uo)) < 2 * tol * np.max(uo)
    su, so = g.stats()[0], o.stats()[0].reshape(ny, nx, 7)
    _, u = o.fields()
    assert np.max(np.abs(su[..., 0] - so[..., 0])) < 2 * nz * tol * np.max(np.abs(u))
    g.close()


@pytest.mark.parametrize("inlet,sponge", [(1, (0, 0.0)), (0, (0, 0.0)), (1, (32, 0.05))])
@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("shape,kernel", [((136, 28, 28), "cell"), ((136, 28, 28), "pair"), ((136, 28, 28), "quad"),
                                          ((136, 28, 28), "staged"), ((132, 30, 28), "quad"), ((132, 30, 28), "auto")])
def test_each_kernel_matches_the_oracle(shape, kernel, precision, inlet, sponge):
    _against_the_oracle(shape, precision, kernel, inlet, sponge)


@pytest.mark.parametrize("inlet", [1, 0])
@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("shape", [(241, 22, 20), (129, 28, 28), (33, 56, 56), (1001, 4, 26), (31, 4, 810)])
def test_odd_lattices_match_the_oracle(shape, precision, inlet):
    _against_the_oracle(shape, precision, "auto", inlet, (0, 0.0))


@pytest.mark.parametrize("inlet", [1, 0])
@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("shape", [(136, 28, 28), (132, 30, 28), (12, 92, 92)])
def test_same_arithmetic_is_bit_identical(shape, precision, inlet):
    got = []
    for kernel in ("pair", "quad", "auto") + (("staged",) if shape[0] % 8 == 0 else ()):
        o, g = _perturbed(shape, precision, kernel, inlet, (shape[0] // 4, 0.05))
        g.step(3)
        got.append((g.populations(), g.utau(), g.stats()[0]))
        g.close()
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("shape,precision", [((128, 32, 32), "fp32"), ((128, 32, 32), "fp16"), ((129, 28, 28), "fp32"),
                                             ((129, 28, 28), "bf16"), ((126, 30, 28), "fp16row")])
def test_graph_periods_and_the_wall_shear_after_them(shape, precision):
    """Periods as graphs (the fork and join of the wall rows among their nodes) give the
    bits of separate launches, and so does the asynchronous wall shear after one."""
    import torch
    from paper_2304_04214_gb300.channel import LBMChannel
    out = []
    for on in (True, False):
        g = LBMChannel(*shape, n_modes=16, seed=21, precision=precision, stats_every=10)
        g.set_graphs(on)
        pinned = torch.empty(2 * g.nx, dtype=torch.float64).pin_memory()
        shear = []
        for n in (192, 1, 127):
            g.step(n)
            g.wall_shear_async(pinned)
            g.sync()
            shear.append(pinned.numpy().copy())
            assert np.array_equal(shear[-1], g.wall_shear().reshape(-1))
        assert g.graph_info()[1] == (3 if on else 0)
        out.append([g.populations(), g.utau(), g.stats()[0], *shear])
        g.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("shape,kernel", [((128, 32, 32), "auto"), ((129, 28, 28), "auto"), ((136, 28, 28), "quad")])
def test_coupling_loop_is_stream_ordered(shape, kernel):
    """A new inlet profile and that step's wall shear every step, without waiting (the
    reduction beside the interior kernel on the side stream, into two pinned buffers in
    turn): the bits of the same loop with a synchronization after every call."""
    import torch
    from paper_2304_04214_gb300.channel import LBMChannel
    runs = []
    for wait in (True, False):
        g = LBMChannel(*shape, n_modes=16, seed=9, step_kernel=kernel)
        U0, R0 = np.empty(g.ny), np.empty(6 * g.ny)
        g.lib.lbm_get_inlet_profile(g.h, _dp(U0), _dp(R0))
        U, R = np.empty_like(U0), np.empty_like(R0)
        bufs = [torch.empty(2 * g.nx, dtype=torch.float64).pin_memory() for _ in range(2)]
        evs = [torch.cuda.Event() for _ in range(2)]
        shear = []
        for n in range(24):
            U[:], R[:] = U0 * (1.0 + 0.02 * np.sin(n)), R0 * (1.0 + 0.05 * np.cos(n))
            assert g.lib.lbm_set_inlet_profile(g.h, _dp(U), _dp(R)) == 0
            g.step(1)
            if wait:
                g.sync()
                shear.append(g.wall_shear().reshape(-1).copy())
                continue
            g.wall_shear_async(bufs[n % 2])
            evs[n % 2].record(g.stream)
            if n:
                evs[(n - 1) % 2].synchronize()
                shear.append(bufs[(n - 1) % 2].numpy().copy())
        if not wait:
            g.sync()
            shear.append(bufs[23 % 2].numpy().copy())
        runs.append([g.populations(), *shear])
        g.close()
    assert len(runs[0]) == len(runs[1]) == 25 and np.max(np.abs(runs[0][-1])) > 0
    for x, y in zip(*runs):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("shape", [(128, 28, 32), (129, 28, 28)])
def test_checkpoint_spacing_does_not_change_the_gradient(shape):
    """Windows whose recomputed steps fork and join the wall rows while the reverse steps
    of the next segment run (even nx), or in line with them (odd nx)."""
    from paper_2304_04214_gb300.channel import LBMChannel
    un = stg_uniforms(16, 27)
    res = []
    for K in (24, 6, 3):
        g = LBMChannel(*shape, n_modes=16, uniforms=un)
        g.step(11)
        J, dJ = g.adjoint_step(24, K, (4, 30, 20))
        res.append((J, dJ, g.adjoint_state_gradient(), g.populations()))
        g.close()
    J0, dJ0, l0, f0 = res[0]
    assert np.any(l0 != 0)
    for J, dJ, lam, f in res[1:]:
        assert abs(J - J0) <= 1e-12 * abs(J0) and np.array_equal(f, f0) and np.array_equal(lam, l0)
        assert np.allclose(dJ, dJ0, rtol=1e-12, atol=0)


@pytest.mark.parametrize("shape,precision,kernel", [
    ((132, 30, 28), "fp16", "quad"),      # a ragged warp
    ((126, 30, 28), "bf16", "auto"),      # four cells a thread, two in the last
    ((132, 30, 28), "fp32", "pair"),
    ((129, 28, 28), "fp32", "auto"),      # odd: interior and wall kernels of one cell
    ((129, 28, 28), "fp16row", "auto"),   # odd: two cells a block's width apart
    ((21, 70, 70), "fp16", "auto"),       # and narrow
    ((1001, 4, 26), "fp32", "auto"),      # wall rows only
])
def test_guard_bands_stay_intact(shape, precision, kernel):
    test_guard_gpu.test_guard_bands_stay_intact(shape, precision, kernel)
