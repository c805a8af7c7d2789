"""Deposit shapes that were set explicitly."""
import statistics

import pytest

import paper_2302_14812_gb300 as rd
from paper_2302_14812_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rd.load_library()


def _dev(tr):
    import torch
    return (torch.from_numpy(tr.x).cuda(), torch.from_numpy(tr.u).cuda(), torch.from_numpy(tr.q).cuda(), tr.t0, tr.dt)


def test_two_cell_shapes_keep_pace():
    """The paired walk takes the same registers in every CTA size: 128 x 2 and 64 x 2 within 7 % of 256 x 2 (13 % apart
    with 96 registers in the smaller ones)."""
    import torch
    tr, det = W.config_undulator(n_part=37, n_steps=3001, n_side=57, n_bins=1021)
    args, shapes = _dev(tr), [(256, 2), (128, 2), (64, 2)]
    d = rd.RadiationDetector.from_workload(det, "mixed")
    ms = {s: [] for s in shapes}
    for _ in range(25):
        for s in shapes:
            d.set_shape(*s)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            d.deposit(*args)
            b.record()
            b.synchronize()
            ms[s].append(a.elapsed_time(b))
    d.close()
    t = {s: statistics.median(v[5:]) for s, v in ms.items()}
    print(t)
    assert t[128, 2] <= 1.07 * t[256, 2] and t[64, 2] <= 1.07 * t[256, 2], t
