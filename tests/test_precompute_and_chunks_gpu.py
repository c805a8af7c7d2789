"""Per-sample precompute at the edges of its 31-sample warp spans, and the default step-chunk rule at its
extremes (one interval, less than its shortest chunk, one CTA's worth, several waves).

Bars: the oracle's (FP64 1e-10, mixed 1e-4)."""
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


def _detector(tr, n_cells, seed=2):
    rng = np.random.default_rng(seed)
    pos = rng.normal(size=(n_cells, 3)) * 20.0
    pos += 25.0 * pos / np.linalg.norm(pos, axis=1, keepdims=True)
    t = tr.t0 + tr.dt * np.arange(tr.n_samples)
    arr = t[None, None] + np.linalg.norm(pos[:, None, None] - tr.x[None], axis=3)
    lo, hi = arr.min() - 0.1, arr.max() + 0.1
    return W.Detector(pos, None, lo, (hi - lo) / 200, 200)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-4)])
@pytest.mark.parametrize("n_part,n_steps,n_cells", [(1, 1, 1), (3, 29, 40), (3, 30, 40), (3, 31, 257), (40, 15, 64),
                                                    (1, 700, 64), (5, 333, 300), (700, 40, 70)])
def test_sizes_around_warp_spans_and_chunks(precision, tol, n_part, n_steps, n_cells):
    import torch
    tr = W.random_smooth(n_part, n_steps, 0.02, max_u=2.0, seed=n_steps)
    det = _detector(tr, n_cells)
    d = rd.RadiationDetector.from_workload(det, precision)
    d.deposit(torch.from_numpy(tr.x).cuda(), torch.from_numpy(tr.u).cuda(), torch.from_numpy(tr.q).cuda(), tr.t0, tr.dt)
    E, B = d.read()
    d.close()
    Eo, Bo, _ = oracle.deposit(tr, det)
    assert parity_err(E, Eo) <= tol and parity_err(B, Bo) <= tol


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("sample", [1, 29, 30, 31, 32, 61, 62, 63])
@pytest.mark.parametrize("what", ["nan", "superluminal"])
def test_a_bad_sample_is_found_at_every_lane(precision, sample, what):
    import torch
    tr = W.random_smooth(2, 63, 0.02, max_u=2.0, seed=1)
    det = _detector(tr, 32)
    x = tr.x.copy()
    if what == "nan":
        x[1, sample, 1] = np.nan
    else:
        x[1, sample:] += 1.0
    d = rd.RadiationDetector.from_workload(det, precision)
    d.deposit(torch.from_numpy(x).cuda(), torch.from_numpy(tr.u).cuda(), torch.from_numpy(tr.q).cuda(), tr.t0, tr.dt)
    with pytest.raises(rd.RDError) as e:
        d.synchronize()
    assert e.value.status == rd.RD_ERR_INPUT
    d.close()
