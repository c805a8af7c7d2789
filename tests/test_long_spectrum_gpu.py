"""Power spectra of long series (columns, then rows) at every split, against numpy's FFT of the same
fields.  Bar: the FP32 transform's 1e-5 of the spectrum tests."""
import numpy as np
import pytest

import paper_2302_14812_gb300 as rd
from parity import parity_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rd.load_library()


@pytest.mark.parametrize("log2n,n_pix", [(14, 3), (14, 341), (15, 2), (16, 5), (17, 43), (18, 2), (19, 1), (20, 2), (21, 2),
                                         (22, 1)])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_long_series(log2n, n_pix, precision):
    """Noise and a few lines in every cell; 341 and 43 cells take a second, shorter batch."""
    n = 1 << log2n
    rng = np.random.default_rng(log2n)
    pos = rng.normal(size=(n_pix, 3)) * 10.0 + 30.0
    d = rd.RadiationDetector(pos, 0.0, 0.03, n, precision=precision)
    t = np.arange(n)
    F = [(0.1 * rng.normal(size=(n_pix, n, 3)) + np.sin(2 * np.pi * rng.integers(1, n // 2, (n_pix, 1, 3)) * t[None, :, None] / n)
          ).astype(np.float32) for _ in range(2)]
    d.write(*F)
    for name, f in zip(("E", "B"), F):
        P = d.power_spectrum(name).cpu().numpy()
        ref = 0.03 ** 2 * np.sum(np.abs(np.fft.rfft(f.astype(np.float64), axis=1)) ** 2, axis=2)
        assert P.shape == ref.shape
        assert parity_err(P, ref) <= 1e-5
    d.close()


def _radix2(x):
    """Stockham radix-2 transform in complex64, roots rounded from FP64."""
    n, s, size = x.shape[-1], 1, x.shape[-1]
    while n > 1:
        i = np.arange(size // 2)
        p, q = i // s, i % s
        w = np.exp(-2j * np.pi * p / n).astype(np.complex64)
        a, b = x[..., : size // 2], x[..., size // 2:]
        y = np.empty_like(x)
        y[..., q + 2 * s * p] = a + b
        y[..., q + 2 * s * p + s] = (a - b) * w
        x, n, s = y, n // 2, 2 * s
    return x


@pytest.mark.parametrize("log2n", [14, 17, 19, 20])
def test_error_no_larger_than_radix2(log2n):
    """The columns-and-rows transform is no less accurate than log2 N radix-2 passes in FP32."""
    n, n_pix = 1 << log2n, 4
    rng = np.random.default_rng(100 + log2n)
    f = rng.normal(size=(n_pix, n, 3)).astype(np.float32)
    d = rd.RadiationDetector(rng.normal(size=(n_pix, 3)) + 30.0, 0.0, 1.0, n, precision="mixed")
    d.write(f, f)
    P = d.power_spectrum("E").cpu().numpy().astype(np.float64)
    d.close()
    ref = np.sum(np.abs(np.fft.rfft(f.astype(np.float64), axis=1)) ** 2, axis=2)
    plain = np.sum(np.abs(_radix2(np.moveaxis(f, 1, 2).astype(np.complex64))[..., : n // 2 + 1].astype(np.complex128)) ** 2,
                   axis=1)
    assert np.linalg.norm(P - ref) <= np.linalg.norm(plain - ref)
