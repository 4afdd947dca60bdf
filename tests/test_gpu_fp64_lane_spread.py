"""FP64 phase models between the launches that the few-orbit kernel takes and
those that fill the GPU: 2 units a lane, on teams of two and four warps past 64
units.  An orbit's bits are those it has among many orbits (4 or 8 units a
lane), for numbers of orbits at both ends of the range and, with checkpoints
kept (the few-orbit kernel then stands aside), for a few; and they are the
oracle's to 1e-12 (the orbit that holds a phase of 2^22, each of whose steps
rounds by 2^-31, to 25 times that, and as much again through the coupling)."""
import numpy as np
import pytest
import torch

import oracle
import paper_1908_03869_gb300 as sdeb
from helpers import max_rel_err, run_oracle
from paper_1908_03869_gb300 import build as sdeb_build
from paper_1908_03869_gb300 import inputs
from paper_1908_03869_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu
STEPS = 25


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    sdeb_build.build()
    sdeb.lib()
    oracle.lib()


def _lines(n):
    """(orbits past the few-orbit kernel's line, orbits that fill the GPU) for n units."""
    lanes = torch.cuda.get_device_properties(0).multi_processor_count * 4 * 2 * 32
    pow2 = 1 << (n - 1).bit_length()
    return lanes // pow2 + 1, -(-lanes // min(32, max(1, pow2 // 4)))


def _inputs(model, n, orbits):
    p, x0 = (inputs.kuramoto if model == "kuramoto" else inputs.kuramoto_paper_speed)(n, 64, seed=n)
    x0[1, 0] = 2.0 ** 22  # phases past both ends of the in-line range
    x0[2, n - 1] = -2.0 ** -13
    x0[3, :] = 0.0
    x0[4, :] = 1e-9 * x0[4, :]
    rep = -(-orbits // 64)
    return np.tile(p, (rep, 1))[:orbits], np.tile(x0, (rep, 1))[:orbits]


def _run(model, n, p, x0, ckpt_every=0):
    """(final states, flags)"""
    pb = sdeb.Problem.make(model, n, len(x0), 0.01, STEPS, STEPS, 3, "fp64", ckpt_every=ckpt_every)
    with Integrator(pb) as it:
        it.set_params(torch.tensor(p, device="cuda"), torch.tensor(x0, device="cuda"))
        it.integrate()
        return it.final().cpu(), it.flags()


@pytest.mark.parametrize("model", ["kuramoto", "kuramoto_paper"])
@pytest.mark.parametrize("n", [3, 4, 7, 8, 15, 31, 32, 33, 63, 65, 100, 128, 129, 130, 200, 255, 256])
def test_bits_between_the_lines(model, n):
    past_few, fills = _lines(n)
    p, x0 = _inputs(model, n, fills)
    many, flags = _run(model, n, p, x0)
    assert not np.asarray(flags).any()
    for orbits in (past_few, (past_few + fills) // 2, fills - 1):
        assert torch.equal(_run(model, n, p[:orbits], x0[:orbits])[0], many[:orbits])
    assert torch.equal(_run(model, n, p[:9], x0[:9], ckpt_every=10)[0], many[:9])
    _, want = run_oracle(model, n, p[:9], x0[:9], 0.01, STEPS, STEPS, seed=3)
    got = many[:9].numpy()
    assert max_rel_err(np.delete(got, 1, 0), np.delete(want, 1, 0)) < 1e-12
    assert np.max(np.abs(got[1] - want[1])) <= 2 * STEPS * 2.0 ** -31


@pytest.mark.parametrize("n", [70, 200])
def test_a_non_finite_orbit_of_a_team_is_flagged_alone(n):
    orbits = _lines(n)[0] + 3
    p, x0 = _inputs("kuramoto", n, orbits)
    clean, _ = _run("kuramoto", n, p, x0)
    x0[7, n - 1] = np.inf
    final, flags = _run("kuramoto", n, p, x0)
    keep = np.arange(orbits) != 7
    assert torch.isnan(final[7]).all() and torch.equal(final[keep], clean[keep])
    assert np.flatnonzero(np.asarray(flags)).tolist() == [7]
