"""A power spectrum of fixed fields is the same bits on every call, at every split of the long series: each
frequency has one writer, also in the two rows that hold both k and N - k."""
import numpy as np
import pytest

import paper_2302_14812_gb300 as rd


def writers(n1, n2):
    """How often the rows 0 .. n1 / 2 of k_split_rows write each frequency 0 .. N / 2."""
    n, half = n1 * n2, n1 // 2
    kk, k2 = np.meshgrid(np.arange(half + 1), np.arange(n2), indexing="ij")
    k = kk + n1 * k2
    k = k[~((k > n // 2) & ((kk == 0) | (kk == half)))]
    return np.bincount(np.where(k <= n // 2, k, n - k), minlength=n // 2 + 1)


@pytest.mark.parametrize("log2n", range(14, 23))
def test_one_writer_per_frequency(log2n):
    """The kernel's index rule, at the splits of split_n2()."""
    n = 1 << log2n
    n2 = 512 if n <= 131072 else min(4096, n // 256)
    assert np.all(writers(n // n2, n2) == 1)


@pytest.mark.gpu
@pytest.mark.parametrize("log2n,n_pix", [(13, 40), (14, 341), (17, 43), (18, 5), (19, 3), (20, 2), (22, 1)])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_same_bits_on_every_call(log2n, n_pix, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 1 << log2n
    g = torch.Generator(device="cuda").manual_seed(log2n)
    f = torch.randn((n_pix, n, 3), generator=g, device="cuda", dtype=torch.float32)
    d = rd.RadiationDetector(np.random.default_rng(1).normal(size=(n_pix, 3)) + 30.0, 0.0, 0.03, n, precision=precision)
    d.write(f, f)
    first = d.power_spectrum("E")
    for _ in range(20):
        assert torch.equal(d.power_spectrum("E"), first)
    d.close()
