"""FP64 phase models whose phases are small: relative precision, the
equilibrium at 0 and mirror symmetry are kept, as sums in FP64 keep them.

Without noise, with K = 1 and equal frequencies, a step moves a phase by a sum of
sines, so everything stays relative to the orbit's largest phase.

Tolerance of the runs: a step of 0.01 rounds its increment, of at most 0.02
of the largest phase, by a few units of 2^-53 and the new phase by one: over
200 steps (four evaluations a step with Runge-Kutta) below 200 (1 + 4 x 0.02 x
8) 2^-53 = 4e-14 of it, on either side; 1e-13 in all.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_1908_03869_gb300 as sdeb
from helpers import run_gpu, run_oracle
from paper_1908_03869_gb300 import build as sdeb_build
from paper_1908_03869_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu
SCHEMES = {"em": {}, "rk4": {"rk4": True}, "midpoint": {"implicit": "midpoint"}}


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    sdeb_build.build()
    sdeb.lib()
    oracle.lib()


def _params(orbits, n):
    p = np.zeros((orbits, n + 2))
    p[:, 0] = 1.0
    return p


@pytest.mark.parametrize("n,scheme", [(n, s) for s in SCHEMES for n in (1, 2, 3, 17, 32, 100, 129, 256)
                                      if s != "midpoint" or n <= 32])  # the oracle solves it densely
def test_relative_to_the_phases(n, scheme):
    scales = np.array([1e-3, 1e-4, 1e-8, 1e-12, 1e-16, 1e-100, 1e-300])
    rng = np.random.default_rng(n)
    x0 = scales[:, None] * rng.uniform(-1.0, 1.0, (len(scales), n))
    _, got = run_gpu("kuramoto", n, _params(len(scales), n), x0, 0.01, 200, 200, **SCHEMES[scheme])
    _, want = run_oracle("kuramoto", n, _params(len(scales), n), x0, 0.01, 200, 200, **SCHEMES[scheme])
    assert np.max(np.abs(got - want) / np.abs(x0).max(1, keepdims=True)) <= 1e-13


@pytest.mark.parametrize("scheme", list(SCHEMES))
@pytest.mark.parametrize("n", [1, 2, 5, 32, 100, 256])
def test_equilibrium_and_mirror_symmetry_are_exact(n, scheme):
    rng = np.random.default_rng(n)
    half = rng.uniform(0.0, 2.0, (3, n // 2)) * np.array([[1.0], [1e-3], [1e-9]])
    mirror = np.concatenate([half, np.zeros((3, n % 2)), -half[:, ::-1]], 1)
    x0 = np.concatenate([np.zeros((1, n)), mirror])
    _, got = run_gpu("kuramoto", n, _params(4, n), x0, 0.01, 50, 50, **SCHEMES[scheme])
    assert not got[0].any()
    if scheme != "midpoint":  # its solve adds FP64 sums in lane order
        assert np.array_equal(got[1:], -got[1:, ::-1])


def test_one_step_moves_by_the_sine_to_its_last_bits():
    """K = n = 2, dt = 1, theta = (x, 0): one step moves the second phase by
    S cos 0 - C sin 0 = sin x, off by 2.25 units of 2^-53 for the sine, one for
    the sum and one for its rounding."""
    rng = np.random.default_rng(2)
    q = np.arange(1, 3000) * (np.pi / 2)
    x = np.concatenate([rng.choice([-1, 1], 20000) * 2.0 ** rng.uniform(-80, 52, 20000), q, np.nextafter(q, 0),
                        q + 2.0 ** rng.uniform(-40, -5, len(q)), [2.0 ** -11, 2.0 ** 21, 2.0 ** 53, 2.0 ** 60]])
    theta = torch.tensor(np.stack([x, np.zeros_like(x)], 1), device="cuda")
    params = torch.tensor([2.0, 0.0, 0.0, 0.0], dtype=torch.float64, device="cuda")
    with Integrator(sdeb.Problem.make("kuramoto", 2, len(x), 1.0, 1, 1, 0, "fp64", shared_params=True)) as it:
        it.set_params(params, theta)
        it.integrate()
        moved = it.final().cpu().numpy()[:, 1]
    exact = np.sin(x.astype(np.longdouble))
    assert np.max(np.abs((moved - exact) / exact)) <= (4.25 + 1.0) * 2.0 ** -53  # the host's own sine: one more
