"""A layout that is asked for is the one that runs, in both precisions and for
any number of orbits (read off the name of the kernel that was launched); a
context left at its default may take other lanes, with the same bits."""
import re

import pytest
import torch

import paper_1908_03869_gb300 as sdeb
from paper_1908_03869_gb300 import build as sdeb_build
from paper_1908_03869_gb300 import inputs
from paper_1908_03869_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    sdeb_build.build()
    sdeb.lib()
    _names(lambda: torch.zeros(8, device="cuda").add_(1.0))  # the profiler's first session may see nothing


def _names(call):
    """Names of the kernels that call launches."""
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    return [e.key for e in prof.key_averages()]


def _run(model, n, orbits, precision, layout):
    """(kernel's lanes per orbit and units per lane, final state)"""
    make = inputs.kuramoto if model == "kuramoto" else inputs.kuramoto_paper_speed
    dtype = torch.float64 if precision == "fp64" else torch.float32
    p, x0 = (torch.tensor(a, dtype=dtype, device="cuda") for a in make(n, orbits, seed=n))
    with Integrator(sdeb.Problem.make(model, n, orbits, 0.01, 10, 10, 3, precision)) as it:
        if layout is not None:
            it.set_layout(*layout)
            assert tuple(it.layout()) == layout
        it.set_params(p, x0)
        names = [k for k in _names(it.integrate) if "em_forward" in k or "em_split" in k]
        assert len(names) == 1
        return re.search(r"(?:float|double), (\d+), (\d+)[,>]", names[0]).groups(), it.final().cpu()


@pytest.mark.parametrize("orbits", [40, 20000])
@pytest.mark.parametrize("model,n,layout", [
    ("kuramoto", 7, (1, 8)), ("kuramoto", 8, (2, 4)), ("kuramoto", 13, (2, 8)), ("kuramoto", 32, (4, 8)),
    ("kuramoto", 32, (8, 4)), ("kuramoto", 60, (4, 16)), ("kuramoto", 128, (8, 16)), ("kuramoto", 100, (32, 4)),
    ("kuramoto", 128, (16, 8)), ("kuramoto", 200, (32, 8)), ("kuramoto_paper", 32, (4, 8)),
    ("kuramoto_paper", 60, (8, 8)), ("kuramoto_paper", 256, (32, 8))])
def test_the_layout_asked_for_runs(model, n, layout, orbits):
    default = _run(model, n, orbits, "fp64", None)[1]
    lanes, final = _run(model, n, orbits, "fp64", layout)
    assert tuple(map(int, lanes)) == layout
    assert torch.equal(final, default)
    lanes, _ = _run(model, n, orbits, "fp32", layout)
    assert tuple(map(int, lanes)) == layout
