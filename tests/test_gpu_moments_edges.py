"""Ensemble moments at the edges of their work split (chunks of 4096 orbits,
rows of 256 threads, groups of 16 elements, lanes per orbit) and of the FP32
pair sums' range, against the moments of the same frames in 64 bits.

Tolerance 1e-13 relative to the state's spread (mean) and to its variance:
4096 elements added in FP64 are off by less than 2^-53 64 = 7e-15 of the sum,
the few dozen merges by a few 2^-53 each.
"""
import numpy as np
import pytest
import torch

import paper_1908_03869_gb300 as sdeb
from paper_1908_03869_gb300 import build as sdeb_build
from paper_1908_03869_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu
DTYPE = {"fp32": torch.float32, "fp64": torch.float64}


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    sdeb_build.build()
    sdeb.lib()


def _moments(model, x0, precision, order=False):
    """(frames, moments, order moments) of one step from x0."""
    orbits, n = x0.shape
    pb = sdeb.Problem.make(model, n, orbits, 1e-3, 1, 1, 0, precision)
    _, d = sdeb.model_shape(model, n)
    p = torch.full((orbits, d), 0.25, dtype=DTYPE[precision], device="cuda")
    with Integrator(pb) as it:
        it.set_params(p, torch.tensor(x0, dtype=DTYPE[precision], device="cuda"))
        it.integrate()
        mom, rmom = it.moments(order_param=order)
        return it.frames().cpu().numpy().astype(np.longdouble), mom.cpu().numpy(), rmom


def _check(fr, mom):
    mean, var = fr.mean(1), fr.var(1)
    assert np.all(np.abs(mom[..., 1] - var) <= 1e-13 * var)
    assert np.all(np.abs(mom[..., 0] - mean) <= 1e-13 * (np.abs(mean) + np.sqrt(var)))


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [1, 2, 7, 33, 100, 255, 256])
@pytest.mark.parametrize("orbits", [2, 17, 300, 4097, 12289])
def test_state_and_order_moments(precision, n, orbits):
    rng = np.random.default_rng(orbits * 1000 + n)
    fr, mom, rmom = _moments("kuramoto", rng.uniform(0, 2 * np.pi, (orbits, n)), precision, order=True)
    _check(fr, mom)
    r = np.hypot(np.cos(fr).mean(2), np.sin(fr).mean(2))
    want = np.stack([r.mean(1), r.var(1)], -1).astype(np.float64)
    np.testing.assert_allclose(rmom.cpu().numpy(), want, rtol=0, atol=1e-6 if precision == "fp32" else 1e-13)


@pytest.mark.parametrize("scale", [1e30, 1e21, 1.0, 1e-10, 1e-20])
@pytest.mark.parametrize("shift", [0.0, 100.0])
def test_scales_past_the_pair_sums(scale, shift):
    rng = np.random.default_rng(5)
    fr, mom, _ = _moments("ou", scale * (shift + rng.standard_normal((4133, 3))) if scale != 1e-20 else
                          scale * (shift + rng.uniform(1, 2, (4133, 3))), "fp32")
    mean, var = fr.mean(1), fr.var(1)
    # the shifted sums lose (mean - first value)^2 / var of the variance at most: 16 / 1 here
    assert np.all(np.abs(mom[..., 1] - var) <= 1e-12 * var)
    assert np.all(np.abs(mom[..., 0] - mean) <= 1e-13 * (np.abs(mean) + np.sqrt(var)))


def test_equal_and_non_finite_elements():
    x0 = np.full((5000, 4), 0.3)
    x0[:, 1] = 0.0
    x0[4500, 2] = np.inf
    x0[10, 3] = np.nan
    pb = sdeb.Problem.make("ou", 4, 5000, 1e-3, 1, 1, 0, "fp32")
    with Integrator(pb) as it:
        it.set_params(torch.zeros((5000, 2), device="cuda"), torch.tensor(x0, dtype=torch.float32, device="cuda"))
        it.integrate()
        mom = it.moments(begin=0, count=1)[0].cpu().numpy()[0]
    assert mom[0, 0] == np.float64(np.float32(0.3)) and mom[0, 1] == 0.0
    assert mom[1, 0] == 0.0 and mom[1, 1] == 0.0
    assert not np.isfinite(mom[2, 0]) and not np.isfinite(mom[3, 0])
