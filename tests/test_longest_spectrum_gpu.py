"""Power spectra of series longer than 2^22 bins (FP64 detectors): radix-2 passes over the whole batch, against the
FP64 transform of the same fields.  Bar: the spectrum tests' 1e-5."""
import numpy as np
import pytest

import paper_2302_14812_gb300 as rd
from parity import parity_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log2n,n_pix", [(23, 1), (23, 3), (24, 1)])
def test_beyond_the_split_lengths(log2n, n_pix):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 1 << log2n
    g = torch.Generator(device="cuda").manual_seed(log2n)
    t = torch.arange(n, device="cuda", dtype=torch.float64)[None, :, None] / n
    d = rd.RadiationDetector(np.random.default_rng(1).normal(size=(n_pix, 3)) + 30.0, 0.0, 0.03, n, precision="fp64")
    F = [(0.1 * torch.randn((n_pix, n, 3), generator=g, device="cuda") +
          torch.sin(2.0 * np.pi * torch.tensor([3.0, 1001.0, n / 5], device="cuda") * t)).float().double() for _ in range(2)]
    d.write(*F)
    for name, f in zip(("E", "B"), F):
        P = d.power_spectrum(name)
        ref = sum(torch.fft.rfft(f[..., i], dim=1).abs().square() for i in range(3)) * 0.03 ** 2
        assert P.shape == ref.shape
        assert parity_err(P.cpu().numpy(), ref.cpu().numpy()) <= 1e-5
        assert torch.equal(P, d.power_spectrum(name))
    d.close()
