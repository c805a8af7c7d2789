"""Streamed deposits of device samples that do not start on an 8-byte boundary (records packed with other data):
the call copies them into place, so the fields are those of aligned samples, bit for bit."""
import numpy as np
import pytest

import paper_2302_14812_gb300 as rd
from paper_2302_14812_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _packed(a, shift):
    """Device bytes holding the float64 array a from byte `shift` on, and its address."""
    import torch
    raw = torch.empty(a.nbytes + 16, dtype=torch.uint8, device="cuda")
    raw[shift:shift + a.nbytes] = torch.from_numpy(np.ascontiguousarray(a).reshape(-1).view(np.uint8)).cuda()
    return raw, raw.data_ptr() + shift


@pytest.mark.parametrize("shifts", [(4, 0, 0), (0, 1, 0), (0, 0, 4), (3, 5, 7)])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_unaligned_samples(precision, shifts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    tr = W.random_smooth(1, 150, 0.02, max_u=2.5, seed=6)
    det = W.Detector(W.spherical_cap(5, 30.0, 0.4), None, 26.0, 0.013, 800)
    got = []
    for shift in ((0, 0, 0), shifts):
        d = rd.RadiationDetector.from_workload(det, precision)
        for a, b in ((0, 1), (1, 60), (60, tr.n_samples)):
            raw, ptr = zip(*(_packed(v, s) for v, s in zip((tr.x[:, a:b], tr.u[:, a:b], tr.q), shift)))
            t = rd.rd_traj()
            t.n_part, t.n_samples, t.mem = 1, b - a, rd.RD_MEM_DEVICE
            t.x, t.u, t.q = ptr
            t.t0, t.dt = tr.t0 + a * tr.dt, tr.dt
            rd.rd_deposit_stream(d.handle, t)
            torch.cuda.synchronize()
            del raw
        got.append(d.read())
        assert d.stats().device_errors == 0
        d.close()
    assert np.abs(got[0][0]).max() > 0
    # one particle, one step chunk a call: at most two partial sums meet in a bin, whose order does not matter
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
