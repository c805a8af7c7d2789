"""Windows that cut arrivals: the tracked walks (bins checked against the window, clipped intervals counted).

Paired walk against the one-cell-per-thread walk, bit for bit (one particle, one step chunk: every bin of a cell is
added once); every interpolation against the oracle (1e-4) with its count of clipped intervals; and the cost of
the tracking, which is a few instructions where a bin edge is passed."""
import statistics

import numpy as np
import pytest

import oracle
import paper_2302_14812_gb300 as rd
from paper_2302_14812_gb300 import workloads as W
from parity import parity_err

pytestmark = pytest.mark.gpu

FULL = rd.RD_NEAR | rd.RD_FAR


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rd.load_library()
    oracle.build()


def _case(n_steps, width, flags, ends):
    """One smooth random motion, 259 cells; ends: bins of the whole window cut off at its start and end, the
    second half of the cells 3 bins later, so that a window's end falls on different intervals."""
    tr = W.random_smooth(1, n_steps, 0.02, max_u=3.0, seed=n_steps)
    rng = np.random.default_rng(n_steps)
    pos = rng.normal(size=(259, 3)) * 20.0
    pos += 25.0 * pos / np.linalg.norm(pos, axis=1, keepdims=True)
    t = tr.t0 + tr.dt * np.arange(tr.n_samples)
    if flags & rd.RD_FARFIELD:
        R = np.linalg.norm(pos, axis=1, keepdims=True)
        arr = t[None] + R - (pos / R) @ tr.x[0].T
    else:
        arr = t[None] + np.linalg.norm(pos[:, None] - tr.x[0][None], axis=2)
    dt_det = width * tr.dt
    first = arr.min(axis=1) - 2.3 * dt_det
    n_bins = int(np.ceil((arr.max(axis=1) - first).max() / dt_det)) + 3
    first = first + (ends[0] + 3.0 * (np.arange(259) % 2)) * dt_det
    return tr, W.Detector(pos, first, 0.0, dt_det, max(1, n_bins - sum(ends)), flags)


def _deposit(tr, det, nc=None):
    import torch
    d = rd.RadiationDetector.from_workload(det, "mixed")
    if nc is not None:
        d.set_shape(128, nc, tr.n_steps, 1)
    d.deposit(torch.from_numpy(tr.x).cuda(), torch.from_numpy(tr.u).cuda(), torch.from_numpy(tr.q).cuda(), tr.t0, tr.dt)
    E, B = d.read("float32")
    st = d.stats()
    d.close()
    assert st.device_errors == 0
    return E, B, st.n_clipped


@pytest.mark.parametrize("ends", [(1, 0), (4, 4), (0, 9)])
@pytest.mark.parametrize("width", [9.0, 2.3, 1.1, 0.45])
@pytest.mark.parametrize("n_steps", [1, 2, 64, 65, 401])
def test_paired_walk_equals_single_steps(n_steps, width, ends):
    tr, det = _case(n_steps, width, FULL, ends)
    E2, B2, c2 = _deposit(tr, det, 2)
    E1, B1, c1 = _deposit(tr, det, 1)
    Eo, Bo, clipped = oracle.deposit(tr, det)
    assert c1 == c2 == clipped
    assert np.array_equal(E2, E1) and np.array_equal(B2, B1)
    assert parity_err(E2, Eo) <= 1e-4 and parity_err(B2, Bo) <= 1e-4


@pytest.mark.parametrize("flags", [FULL | rd.RD_LINEAR, FULL | rd.RD_HOLD_PREV, FULL | rd.RD_QUADRATIC,
                                   rd.RD_FAR | rd.RD_FARFIELD, rd.RD_FAR | rd.RD_FARFIELD | rd.RD_LINEAR,
                                   rd.RD_FAR | rd.RD_FARFIELD | rd.RD_QUADRATIC])
@pytest.mark.parametrize("ends", [(4, 4), (0, 9)])
@pytest.mark.parametrize("width", [9.0, 1.1, 0.45])
@pytest.mark.parametrize("n_steps", [2, 65, 130])
def test_every_walk_in_a_cut_window(n_steps, width, ends, flags):
    tr, det = _case(n_steps, width, flags, ends)
    E, B, c = _deposit(tr, det)
    Eo, Bo, clipped = oracle.deposit(tr, det)
    assert c == clipped
    assert parity_err(E, Eo) <= 1e-4 and parity_err(B, Bo) <= 1e-4


@pytest.mark.parametrize("interp", [rd.RD_LINEAR, rd.RD_HOLD_PREV, rd.RD_QUADRATIC])
def test_cost_of_a_cut_window(interp):
    """An undulator run whose window leaves out a quarter of the arrival span at each end takes no more than 1.25
    times the whole window's time (with every cut chunk walked interval by interval, cell by cell: 1.4)."""
    import torch
    tr, det = W.config_undulator(n_part=100, n_steps=1500, n_side=100, n_bins=1500)
    tr.x, tr.u, tr.q = (torch.from_numpy(a).cuda() for a in (tr.x, tr.u, tr.q))
    cut = det.n_bins // 4
    dets = [rd.RadiationDetector(det.pix_pos, det.t_min + n * det.dt_det, det.dt_det, det.n_bins - 2 * n, det.pix_t0,
                                 flags=FULL | interp) for n in (0, cut)]
    ms = [[], []]
    for _ in range(12):
        for d, out in zip(dets, ms):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            d.deposit(tr.x, tr.u, tr.q, tr.t0, tr.dt)
            b.record()
            b.synchronize()
            out.append(a.elapsed_time(b))
    assert dets[1].stats().n_clipped > 0
    for d in dets:
        d.close()
    whole, part = (statistics.median(m[3:]) for m in ms)
    print(f"whole window {whole:.3f} ms, cut {part:.3f} ms")
    assert part <= 1.25 * whole, (whole, part)
