"""Streamed deposits at the largest calls: one particle with more samples than a 32-bit count of coordinates
holds.  The streamed call stages the samples and then deposits as one call on the whole trajectory does, so the
fields must be the same bits."""
import numpy as np
import pytest

import paper_2302_14812_gb300 as rd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("have", [0, 1])
def test_more_coordinates_than_int32(have):
    """3 m = 2^31 + 1 coordinates in one call; have: a first call of one sample before it.  The window holds the
    arrivals of the last 600 samples."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.mem_get_info()[0] < 150e9:
        pytest.skip("needs 150 GB of free device memory")
    m, dt, dist = 715_827_883, 2.0 ** -10, 50.0
    n = m + have
    x = torch.zeros((1, n, 3), dtype=torch.float64, device="cuda")
    for a in range(0, n, 1 << 26):                              # along z, at a tenth of the speed of light
        b = min(n, a + (1 << 26))
        x[0, a:b, 2] = 0.1 * dt * torch.arange(a, b, dtype=torch.float64, device="cuda")
    u = torch.zeros((1, n, 3), dtype=torch.float64, device="cuda")
    u[0, :, 2] = 0.1 / np.sqrt(1.0 - 0.01)
    end = 0.1 * dt * (n - 1)
    pos = np.array([[0.0, dist, end], [dist, 0.0, end + 3.0]])
    arr = dt * (n - 1) + np.array([dist, np.hypot(dist, 3.0)])
    dt_det = 10.0 * dt
    got = []
    for streamed in (False, True):
        d = rd.RadiationDetector(pos, 0.0, dt_det, 64, arr - 61.3 * dt_det)
        if streamed:
            if have:
                d.deposit_stream(x[:, :have].contiguous(), u[:, :have].contiguous(), None, 0.0, dt)
            d.deposit_stream(x[:, have:], u[:, have:], None, have * dt, dt)
        else:
            d.deposit(x, u, None, 0.0, dt)
        got.append(d.read("float64"))
        assert d.stats().device_errors == 0
        d.close()
    assert np.all(np.abs(got[0][0]).sum(axis=2)[:, 5:60] > 0)
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
