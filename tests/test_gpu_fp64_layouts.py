"""FP64 phase models: the coupling sums are exact integers, so an orbit has
the same bits on every layout its kernel can run on -- few orbits (2 units a
lane, teams of warps past 64 units) and many (4 or 8 units a lane)."""
import pytest
import torch

import paper_1908_03869_gb300 as sdeb
from paper_1908_03869_gb300 import inputs
from paper_1908_03869_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu

MANY_LANES = 152 * 4 * 2 * 32  # from here on 4 units a lane


def _final(model, n, p, x0, layout=None):
    pb = sdeb.Problem.make(model, n, len(x0), 0.01, 25, 25, 3, "fp64")
    with Integrator(pb) as it:
        it.set_params(torch.tensor(p, device="cuda"), torch.tensor(x0, device="cuda"))
        if layout:
            it.set_layout(*layout)
        it.integrate()
        return it.final().cpu()


@pytest.mark.parametrize("model", ["kuramoto", "kuramoto_paper"])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 8, 15, 17, 32, 33, 64, 65, 100, 128, 129, 200, 256])
def test_few_orbits_have_the_bits_of_many(model, n):
    few, many = 7, MANY_LANES // max(1, n // 8) + 5
    p, x0 = (inputs.kuramoto if model == "kuramoto" else inputs.kuramoto_paper_speed)(n, many, seed=n)
    x0[1, 0] = 2.0 ** 22  # phases past both ends of the fixed-point range
    x0[2, n - 1] = -2.0 ** -13
    x0[3, :] = 0.0
    many_final = _final(model, n, p, x0)
    assert torch.isfinite(many_final).all()
    assert torch.equal(many_final[:few], _final(model, n, p[:few], x0[:few]))
    if model == "kuramoto" and 8 < n <= 128:
        assert torch.equal(many_final[:few], _final(model, n, p[:few], x0[:few], (32, 4)))


@pytest.mark.parametrize("n", [4, 40, 100, 200])
def test_a_non_finite_phase_takes_its_orbit_alone(n):
    p, x0 = inputs.kuramoto(n, 9, seed=n)
    clean = _final("kuramoto", n, p, x0)
    x0[4, n // 2] = float("inf")
    final = _final("kuramoto", n, p, x0)
    assert torch.isnan(final[4]).all()
    keep = [0, 1, 2, 3, 5, 6, 7, 8]
    assert torch.equal(final[keep], clean[keep])
