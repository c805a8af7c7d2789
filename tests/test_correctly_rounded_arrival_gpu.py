"""The FP64 deposit's arrival times at distances whose square root lies within 2^-45 of a rounding boundary (in
units of the last place): the correctly rounded root, as the oracle's.

A bin is 128 units in the last place of the distance wide and the interval crosses a bin edge, so that one unit
moves 3 % of a bin's value; bar: the FP64 path's 1e-10."""
import math

import numpy as np
import pytest

import oracle
import paper_2302_14812_gb300 as rd
from paper_2302_14812_gb300 import workloads as W
from parity import parity_err

pytestmark = pytest.mark.gpu


def hard_squares(n):
    """FP64 numbers a in [1, 4) whose roots lie |r| / (4 m) units from a midpoint: 4 a 2^104 = m^2 - r with m odd
    and 2^55 | m^2 - r, for small r = 1 mod 8 (such r have square roots modulo any power of two)."""
    out, i = [], 0
    while len(out) < n:
        r = 1 + 8 * ((i + 1) // 2) * (1 if i % 2 else -1)
        i += 1
        m = 1
        for b in range(3, 56):                  # lift the root of r from modulo 2^b to 2^(b+1)
            if (m * m - r) % (1 << (b + 1)):
                m += 1 << (b - 1)
        assert (m * m - r) % (1 << 55) == 0
        for root in (m, -m, m + (1 << 54), (1 << 54) - m):
            root %= 1 << 55
            if (1 << 53) < root < (1 << 54):
                a = (root * root - r) // 4
                # the square in 53 bits; its correctly rounded root in units of 2^-52
                assert a % (1 << max(0, a.bit_length() - 53)) == 0
                out.append((math.ldexp(float(a), -104), (root - 1) // 2 if r > 0 else (root + 1) // 2))
    return out[:n]


def legs(a):
    """x, y with fl(fl(x x) + fl(y y)) = a."""
    x = math.sqrt(a)
    while x * x > a:
        x = math.nextafter(x, 0.0)
    y = math.sqrt(a - x * x)
    assert x * x + y * y == a
    return x, y


def test_hard_distances():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    oracle.build()
    cases = hard_squares(600)
    pos = np.array([(*legs(a), 0.0) for a, _ in cases])
    R = np.array([math.ldexp(float(k), -52) for _, k in cases])
    assert np.array_equal(np.sqrt([a for a, _ in cases]), R)
    dt_det, dt = 2.0 ** -45, 2.0 ** -46
    x = np.zeros((1, 2, 3))
    tr = W.Trajectories(x, np.zeros_like(x), np.ones(1), 0.0, dt)
    det = W.Detector(pos, R - 1.75 * dt_det, 0.0, dt_det, 8)
    Eo, _, _ = oracle.deposit(tr, det)
    d = rd.RadiationDetector.from_workload(det, "fp64")
    d.deposit(torch.from_numpy(tr.x).cuda(), torch.from_numpy(tr.u).cuda(), torch.from_numpy(tr.q).cuda(), tr.t0, tr.dt)
    E, _ = d.read()
    d.close()
    assert np.count_nonzero(np.abs(Eo).sum(axis=2)) == 2 * len(cases)
    assert parity_err(E, Eo) <= 1e-10
