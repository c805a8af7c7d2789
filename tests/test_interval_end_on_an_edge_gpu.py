"""Intervals of the mixed deposit that end on a bin edge to the last digit, two edges on: the arrival time is
twice the bin width W (in steps) exactly, and W is chosen so that 2 W times the rounded 1 / W falls below 2.

A charge at rest has arrivals one step apart, so the last interval of a trajectory passes two edges for 1/2 < W
< 1, and the time origin puts its end on an edge.  Bar: the oracle's for the mixed path, 1e-4."""
import numpy as np
import pytest

import oracle
import paper_2302_14812_gb300 as rd
from paper_2302_14812_gb300 import workloads as W
from parity import parity_err

pytestmark = pytest.mark.gpu

HELD = rd.RD_NEAR | rd.RD_FAR


def _widths():
    """Bin widths in (1/2, 1), FP32 numbers, for which fl(2 W fl(1 / W)) < 2."""
    w = np.linspace(0.55, 0.97, 400).astype(np.float32)
    w = w[(np.float32(2) * w) * (np.float32(1) / w) < np.float32(2)]
    return [float(v) for v in w[np.linspace(0, len(w) - 1, 4).astype(int)]]


@pytest.mark.parametrize("cut", [False, True])
@pytest.mark.parametrize("n_steps", [1, 2, 64, 65])
@pytest.mark.parametrize("width", _widths())
@pytest.mark.parametrize("flags,shape", [(HELD, None), (HELD, (128, 1)), (HELD, (128, 2)), (HELD | rd.RD_LINEAR, None)])
def test_last_interval_ends_two_edges_on(width, n_steps, cut, flags, shape):
    """cut: the window ends at that edge."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    oracle.build()
    dt, dist, n_pix = 0.5, 10.0, 70
    dt_det = width * dt
    x = np.zeros((1, n_steps + 1, 3))
    tr = W.Trajectories(x, np.zeros_like(x), np.ones(1), 0.0, dt)
    pos = np.random.default_rng(2).normal(size=(n_pix, 3))
    pos *= dist / np.linalg.norm(pos, axis=1, keepdims=True)
    edge = int(np.ceil(n_steps / width)) + 3
    t_min = n_steps * dt + dist - (edge + 1e-9) * dt_det
    det = W.Detector(pos, None, t_min, dt_det, edge if cut else edge + 3, flags)
    d = rd.RadiationDetector.from_workload(det, "mixed")
    if shape is not None:
        d.set_shape(*shape)
    d.deposit(torch.from_numpy(tr.x).cuda(), torch.from_numpy(tr.u).cuda(), torch.from_numpy(tr.q).cuda(), tr.t0, tr.dt)
    E, B = d.read()
    d.close()
    Eo, Bo, _ = oracle.deposit(tr, det)
    assert parity_err(E, Eo) <= 1e-4
    assert np.abs(B).max() <= 1e-5 * np.abs(E).max()        # a charge at rest: E along n
