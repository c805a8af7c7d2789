"""The FP64 deposit in units that take its square root and reciprocal out of FP32's range: lengths and times
scaled by a power of two, which scales every field by its inverse square exactly.

Bar: the scaled run may differ by rounding only where the two forms round differently (1 ulp of R and of
1/(kappa R), amplified by gamma^2 ~ 10 in kappa): 1e-13 of the fields' norm."""
import numpy as np
import pytest

import paper_2302_14812_gb300 as rd
from paper_2302_14812_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(tr, det, scale):
    import torch
    pos = det.pix_pos * scale
    t0 = None if det.pix_t0 is None else det.pix_t0 * scale
    d = rd.RadiationDetector(pos, det.t_min * scale, det.dt_det * scale, det.n_bins, t0, "fp64", det.flags)
    d.deposit(torch.from_numpy(tr.x * scale).cuda(), torch.from_numpy(tr.u).cuda(), torch.from_numpy(tr.q).cuda(),
              tr.t0 * scale, tr.dt * scale)
    E, B = d.read()
    st = d.stats()
    d.close()
    assert st.device_errors == 0
    return E * scale ** 2, B * scale ** 2


@pytest.mark.parametrize("power", [-170, -60, 45, 170])
@pytest.mark.parametrize("flags", [rd.RD_NEAR | rd.RD_FAR, rd.RD_NEAR | rd.RD_FAR | rd.RD_LINEAR])
def test_scaled_units(power, flags):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    tr = W.random_smooth(2, 90, 0.02, max_u=3.0, seed=3)
    rng = np.random.default_rng(3)
    pos = rng.normal(size=(70, 3)) * 20.0
    pos += 25.0 * pos / np.linalg.norm(pos, axis=1, keepdims=True)
    det = W.Detector(pos, np.linalg.norm(pos, axis=1) - 5.0, 0.0, 0.03, 400, flags)
    E0, B0 = _run(tr, det, 1.0)
    E, B = _run(tr, det, 2.0 ** power)
    assert np.linalg.norm(E - E0) <= 1e-13 * np.linalg.norm(E0) and np.linalg.norm(E0) > 0
    assert np.linalg.norm(B - B0) <= 1e-13 * np.linalg.norm(B0)
