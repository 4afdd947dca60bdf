"""Sine and cosine of the FP64 path (64-bit fixed point) at the edges of its
range, read off one step of two coupled phases.

With K = n = 2, dt = 1, sigma = omega = 0 and theta = (x, y), one step moves
y by S cos y - C sin y = sin(x - y) expanded in the sums: y = 0 gives
sin x, y = float(-pi/2) gives cos x + cos(y) sin x with cos(y) = 6e-17.
"""
import math

import numpy as np
import pytest
import torch

import paper_1908_03869_gb300 as sdeb
from paper_1908_03869_gb300 import build
from paper_1908_03869_gb300.integrator import Integrator

# The value itself is within 0.6 units of 2^-53 of the exact one, libm's
# within 1, and the step's sums and its state round a few times at most 1.
TOL = 8 * 2.0 ** -53


def _phases(kind):
    g = np.random.Generator(np.random.PCG64(3))
    if kind == "range_ends":
        e = np.array([2.0 ** -11, 2.0 ** 21])
        x = np.concatenate([e, np.nextafter(e, 0), np.nextafter(e, 1e9), 2.0 ** np.arange(-60, 30.0)])
    elif kind == "quarter_turns":
        q = np.arange(0, 4000) * (math.pi / 2)
        x = np.concatenate([q, np.nextafter(q, 1e9), q + 2.0 ** -30, q - 2.0 ** -45])
    elif kind == "table_steps":
        q = np.arange(0, 1700) / 256.0
        x = np.concatenate([q, np.nextafter(q, 1e9), np.nextafter(q, -1)])
    else:
        x = g.uniform(-1, 1, 8000) * 2.0 ** g.uniform(-14, 24, 8000)
    return np.concatenate([x, -x])


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["range_ends", "quarter_turns", "table_steps", "all_sizes"])
@pytest.mark.parametrize("second,of", [(0.0, math.sin), (-math.pi / 2, math.cos)])
def test_sine_and_cosine(kind, second, of):
    x = _phases(kind)
    theta = torch.tensor(np.stack([x, np.full_like(x, second)], 1), device="cuda")
    params = torch.tensor([2.0, 0.0, 0.0, 0.0], dtype=torch.float64, device="cuda")
    pb = sdeb.Problem.make("kuramoto", 2, len(x), 1.0, 1, 1, 0, "fp64", shared_params=True)
    with Integrator(pb) as it:
        it.set_params(params, theta)
        it.integrate()
        moved = it.final().cpu().numpy()[:, 1] - second
    exact = np.array([of(float(v)) for v in x])
    assert np.max(np.abs(moved - exact)) <= TOL


@pytest.mark.gpu
@pytest.mark.parametrize("bad", [math.inf, -math.inf, math.nan])
def test_non_finite_phase_is_flagged(bad):
    theta = torch.tensor([[bad, 1.0], [2.0, 1.0]], dtype=torch.float64, device="cuda")
    params = torch.tensor([2.0, 0.0, 0.0, 0.0], dtype=torch.float64, device="cuda")
    with Integrator(sdeb.Problem.make("kuramoto", 2, 2, 0.1, 3, 1, 0, "fp64", shared_params=True)) as it:
        it.set_params(params, theta)
        it.integrate()
        final = it.final().cpu().numpy()
        assert it.flags().tolist() == [1, 0]
    assert np.isnan(final[0]).any() and np.isfinite(final[1]).all()


def test_tables():
    trig, log = build.fixed_tables()
    assert len(trig) == 403 and 402 / 256 < math.pi / 2 < 403 / 256
    for j, (c, s) in enumerate(trig):
        assert abs(c / 2 ** 62 - math.cos(j / 256)) < 1e-15 and abs(s / 2 ** 62 - math.sin(j / 256)) < 1e-15
    for j, (lnc, c) in enumerate(log):
        assert c < 2 ** 16 and c * (257 + j) <= 512 << 15 < (c + 1) * (257 + j)
        assert abs(lnc / 2 ** 58 - math.log(c / 2 ** 15)) < 1e-15
    assert log[255] == (0, 1 << 15)
