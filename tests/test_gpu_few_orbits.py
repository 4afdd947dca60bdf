"""The few-orbit kernel (noise on warps of its own) gives the bits of the
kernel that many orbits take: an orbit alone against the same orbit among
enough others to fill the GPU, at the edges of the kernel's lane groups and
of its buffers of eight steps, whole and in ranges, with frames and flags.
"""
import pytest
import torch

import paper_1908_03869_gb300 as sdeb
from paper_1908_03869_gb300 import build as sdeb_build
from paper_1908_03869_gb300 import inputs
from paper_1908_03869_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu
FILLS = 152 * 4 * 32 * 2 + 33  # orbits past the kernel's line for every n


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    sdeb_build.build()
    sdeb.lib()


def _run(model, n, p, x0, precision, steps, stride, ranges=()):
    dtype = torch.float64 if precision == "fp64" else torch.float32
    pb = sdeb.Problem.make(model, n, len(x0), 0.01, steps, stride, 3, precision)
    with Integrator(pb) as it:
        it.set_params(p.to(dtype).cuda(), x0.to(dtype).cuda())
        k = 0
        for end in (*ranges, steps):
            it.integrate_range(k, end)
            k = end
        return it.frames().cpu(), it.final().cpu(), it.flags()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("model", ["kuramoto", "kuramoto_paper"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 32, 33, 64, 65, 100, 128, 129, 256])
def test_bits_of_the_many_orbit_kernel(model, n, precision):
    make = inputs.kuramoto if model == "kuramoto" else inputs.kuramoto_paper_speed
    few, steps = 37, 27
    p, x0 = (torch.tensor(a) for a in make(n, 211, seed=n))
    rep = -(-FILLS // 211)
    many = _run(model, n, p.repeat(rep, 1), x0.repeat(rep, 1), precision, steps, 9)
    for ranges in ((), (8, 9, 25)):
        got = _run(model, n, p[:few], x0[:few], precision, steps, 9, ranges)
        assert torch.equal(got[0], many[0][:, :few]) and torch.equal(got[1], many[1][:few])
        assert not got[2].any()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [3, 20, 70])
def test_a_non_finite_orbit_is_flagged_alone(n, precision):
    p, x0 = (torch.tensor(a) for a in inputs.kuramoto(n, 9, seed=n))
    clean = _run("kuramoto", n, p, x0, precision, 20, 20)
    x0[4, n // 2] = float("nan")
    _, final, flags = _run("kuramoto", n, p, x0, precision, 20, 20)
    keep = [0, 1, 2, 3, 5, 6, 7, 8]
    assert torch.equal(final[keep], clean[1][keep])
    assert flags.tolist() == [0, 0, 0, 0, 1, 0, 0, 0, 0]
