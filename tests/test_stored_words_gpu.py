"""The stored words themselves (the bound device memory) after set_populations, and what
populations reads from them: the two conversions apart, to the rounding of a word."""
import numpy as np
import pytest

from gpu_helpers import bf16_row_base, make_pair
from oracle.oracle import cell_api
from paper_2304_04214_gb300.inputs import noise

pytestmark = pytest.mark.gpu

BITS = {"fp32": 24, "fp16": 11, "bf16": 8, "fp16row": 11}           # significant bits of a word


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _words(g):
    """The current lattice's words as FP64, [19][nz][ny][nx] (the first lattice starts the memory)."""
    import torch
    t = {"fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16, "fp16row": torch.float16}[g.precision]
    assert g.time == 0
    n = 19 * g.ncell * t.itemsize
    return g.mem[:n].view(t).double().cpu().numpy().reshape(19, g.nz, g.ny, g.nx)


@pytest.mark.parametrize("precision", list(BITS))
@pytest.mark.parametrize("shape", [(3, 4, 1), (33, 6, 5), (64, 16, 9), (129, 12, 7)])
def test_words_and_the_values_read_from_them(shape, precision):
    """A word is within half of its last place of the value it holds (f, f - w, or f - w -
    base(j)), and populations within the FP32 rounding of word + base of what the words
    say.  The library forms the base (below 2^-6) in FP64 and stores it in FP32, as here:
    their last place, 2^-30, is all that may differ."""
    nx, ny, nz = shape
    o, g = make_pair(nx, ny, nz, n_modes=4, precision=precision)
    f = o.state() * (1.0 + 0.02 * noise((19, nz, ny, nx), seed=5))
    w = cell_api.matrix()[1][:, None, None, None]
    base = bf16_row_base(o).astype(np.float64)[:, None, :, None]
    ref = np.zeros_like(w) if precision == "fp32" else w if precision == "fp16" else w + base
    last = 0.0 if precision in ("fp32", "fp16") else 2.0 ** -30
    assert np.max(np.abs(base)) < 2.0 ** -6
    g.set_populations(f)
    words, dev = _words(g), f - ref
    half = 2.0 ** -BITS[precision] * np.abs(dev)
    if precision in ("fp16", "fp16row"):
        half = np.maximum(half, 2.0 ** -25)                         # below 2^-14: half of the smallest word
    assert np.all(np.abs(words - dev) <= half + last + 2.0 ** -24 * np.abs(dev))
    # the rounding is less than the change of the base from row to row and than the noise
    assert precision == "fp32" or np.max(half) < 0.1 * np.max(np.abs(0.02 * f))
    got = g.populations()
    said = words + ref
    assert np.all(np.abs(got - said) <= 2.0 ** -24 * np.abs(said - w) + last + 2.0 ** -52)
    if precision in ("fp32", "fp16"):
        assert np.array_equal(got, said)
    g.close()
