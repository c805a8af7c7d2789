"""The paired walk of the mixed deposit (two cells per thread, two intervals per crossing update).

The one-cell-per-thread shape walks the same operations one interval at a time, and one particle in one
step chunk adds every (cell, bin) once, so the two shapes must give the same FP32 fields, bit for bit.
The bin widths (in steps) cover: two intervals that seldom pass an edge, that pass one in either
interval, that pass one each (the single-step fallback), and intervals that pass several (the exact
walk).  The lengths cover odd and even step counts around a 64-interval tile and its neighbours.
"""
import numpy as np
import pytest

import oracle
import paper_2302_14812_gb300 as rd
from paper_2302_14812_gb300 import workloads as W
from parity import parity_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rd.load_library()
    oracle.build()


def _case(n_steps, width, flags=rd.RD_NEAR | rd.RD_FAR):
    """One smooth random motion, 259 cells (a ragged second block), a window around every arrival."""
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
    return tr, W.Detector(pos, first, 0.0, dt_det, n_bins, flags)


def _deposit(tr, det, nc=None):
    import torch
    d = rd.RadiationDetector.from_workload(det, "mixed")
    if nc is not None:
        d.set_shape(128, nc, tr.n_steps, 1)     # (a small grid of the default 256 x 2 runs one cell per thread)
    d.deposit(torch.from_numpy(tr.x).cuda(), torch.from_numpy(tr.u).cuda(), torch.from_numpy(tr.q).cuda(), tr.t0, tr.dt)
    E, B = d.read("float32")
    st = d.stats()
    d.close()
    assert st.device_errors == 0 and st.n_clipped == 0
    return E, B


@pytest.mark.parametrize("width", [9.0, 2.3, 1.1, 0.45, 0.1])
@pytest.mark.parametrize("n_steps", [1, 2, 3, 63, 64, 65, 66, 130, 401])
def test_paired_walk_equals_single_steps(n_steps, width):
    tr, det = _case(n_steps, width)
    E2, B2 = _deposit(tr, det, 2)
    E1, B1 = _deposit(tr, det, 1)
    assert np.array_equal(E2, E1) and np.array_equal(B2, B1)
    Eo, Bo, _ = oracle.deposit(tr, det)
    assert parity_err(E2, Eo) <= 1e-4 and parity_err(B2, Bo) <= 1e-4


@pytest.mark.parametrize("width", [9.0, 1.1, 0.45])
@pytest.mark.parametrize("n_steps", [2, 65, 130])
def test_paired_walk_in_the_far_field_limit(n_steps, width):
    tr, det = _case(n_steps, width, rd.RD_FAR | rd.RD_FARFIELD)
    E, B = _deposit(tr, det)
    Eo, Bo, _ = oracle.deposit(tr, det)
    assert parity_err(E, Eo) <= 1e-4 and parity_err(B, Bo) <= 1e-4


@pytest.mark.parametrize("flags", [rd.RD_NEAR | rd.RD_FAR, rd.RD_FAR | rd.RD_FARFIELD])
@pytest.mark.parametrize("width", [0.45, 0.1, 0.03])
@pytest.mark.parametrize("n_steps", [1, 65, 130])
def test_runs_of_bins(n_steps, width, flags):
    """Intervals of 1 to 60 bins: short runs lane by lane, long ones handed over to groups of lanes; whole
    windows, and windows that begin and end inside runs (clipping)."""
    tr, det = _case(n_steps, width, flags)
    E, B = _deposit(tr, det)
    Eo, Bo, _ = oracle.deposit(tr, det)
    assert parity_err(E, Eo) <= 1e-4 and parity_err(B, Bo) <= 1e-4
    cut = W.Detector(det.pix_pos, det.pix_t0 + 7.4 * det.dt_det, 0.0, det.dt_det, max(1, det.n_bins - 16), flags)
    Eo, Bo, clipped = oracle.deposit(tr, cut)
    import torch
    d = rd.RadiationDetector.from_workload(cut, "mixed")
    d.deposit(torch.from_numpy(tr.x).cuda(), torch.from_numpy(tr.u).cuda(), torch.from_numpy(tr.q).cuda(), tr.t0, tr.dt)
    E, B = d.read()
    st = d.stats()
    d.close()
    assert st.n_clipped == clipped and st.device_errors == 0
    assert parity_err(E, Eo) <= 1e-4 and parity_err(B, Bo) <= 1e-4


@pytest.mark.parametrize("n_cells", [1, 63, 64, 65, 256, 257, 700])
def test_small_grids_run_one_cell_per_thread(n_cells):
    """The default shape on a small grid against the two-cell shape it stands in for."""
    tr, det = _case(130, 1.1)
    det = W.Detector(np.resize(det.pix_pos, (n_cells, 3)), np.resize(det.pix_t0, n_cells), 0.0, det.dt_det, det.n_bins)
    E2, B2 = _deposit(tr, det, 2)
    import torch
    d = rd.RadiationDetector.from_workload(det, "mixed")
    d.set_chunk(tr.n_steps)
    d.deposit(torch.from_numpy(tr.x).cuda(), torch.from_numpy(tr.u).cuda(), torch.from_numpy(tr.q).cuda(), tr.t0, tr.dt)
    E, B = d.read("float32")
    d.close()
    assert np.array_equal(E, E2) and np.array_equal(B, B2)
