"""Populations between host FP64 arrays and the stored words, converted on the
device a chunk at a time: every storage, lattices whose chunks end anywhere."""
import numpy as np
import pytest

from gpu_helpers import make_pair, quantize_state
from paper_2304_04214_gb300.inputs import noise

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16", "fp16row"])
@pytest.mark.parametrize("shape", [(3, 4, 1), (33, 6, 5), (64, 16, 9)])
def test_populations_round_trip_by_the_storage_rule(shape, precision):
    """set rounds as quantize_state does (the NumPy statement of the storage),
    get returns exactly that; a second round trip changes nothing.  (FP32
    addition of word and base: exact in quantize_state's FP32 arithmetic.)"""
    nx, ny, nz = shape
    o, g = make_pair(nx, ny, nz, n_modes=4, precision=precision)
    f = o.state() * (1.0 + 0.02 * noise((19, nz, ny, nx), seed=5))
    want = quantize_state(f, precision, o)
    g.set_populations(f)
    got = g.populations()
    if precision in ("fp32", "fp16"):
        assert np.array_equal(got, want)
    else:                                        # the library's FP32 row base may differ in its last bit
        assert np.max(np.abs(got - want)) <= (2.0 ** -8 if precision == "bf16" else 2.0 ** -11) * np.max(np.abs(f))
    g.set_populations(got)
    assert np.array_equal(g.populations(), got)
