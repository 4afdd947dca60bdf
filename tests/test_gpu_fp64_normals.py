"""FP64 normals relative to themselves, at the edges of the logarithm's and the
angle's ranges: the radius word next to 0 and to 2^32 and on both sides of the
logarithm's table steps, the angle word next to multiples of a quarter turn,
found among four million blocks.

Bounds in units of 2^-53: three (a radius half a unit off before it is rounded,
a sine 1.1, the product's rounding 1); within 2^-14 of a multiple of a quarter
turn the small one may be the product of the rounded radius (1.5) with CUDA's
sincospi (two units in the last place: 4) and its rounding: 6.5.  One more for
the host's own logarithm and sine.
"""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_1908_03869_gb300 as sdeb
from paper_1908_03869_gb300 import build as sdeb_build

pytestmark = pytest.mark.gpu
STEPS, ORBITS = 1024, 4096


@pytest.fixture(scope="module")
def blocks():
    """(words [.., 2], normals [.., 2]) of the word pairs worth looking at."""
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    sdeb_build.build()
    sdeb.lib()
    oracle.lib()
    z = torch.empty((STEPS, ORBITS, 4), dtype=torch.float64, device="cuda")
    sdeb.sdeb_normals_fill(5, 0, STEPS, 0, ORBITS, 4, sdeb.SDEB_FP64, ctypes.c_void_p(z.data_ptr()))
    w = oracle.philox_fill(5, 0, STEPS, 0, 1, 0, ORBITS)[:, 0]
    return w.reshape(-1, 2).astype(np.uint64), z.cpu().numpy().reshape(-1, 2)


def _exact(w):
    one = np.longdouble(1)
    u = (w[:, 0].astype(np.longdouble) + 0.5) / 2 ** 32
    from_one = (2.0 ** 32 - 0.5 - w[:, 0].astype(np.longdouble)) / 2 ** 32  # 1 - u, exact
    r = np.sqrt(-2 * np.where(u > 0.5, np.log1p(-from_one), np.log(u)))
    t = 2 * w[:, 1] + 1  # 33 bits of a turn
    f = (t & np.uint64(2 ** 31 - 1)).astype(np.longdouble) / 2 ** 31  # of the quadrant
    half_pi = 2 * np.arctan(one)
    s = np.where(f <= 0.5, np.sin(half_pi * f), np.cos(half_pi * (1 - f)))
    c = np.where(f <= 0.5, np.cos(half_pi * f), np.sin(half_pi * (1 - f)))
    q = (t >> np.uint64(31)).astype(int)
    cos, sin = np.choose(q, [c, -s, -c, s]), np.choose(q, [s, c, -s, -c])
    near = np.minimum(f, 1 - f) * half_pi < 2.0 ** -14
    return np.stack([r * cos, r * sin], 1), near


def _check(w, z):
    want, near = _exact(w)
    units = np.max(np.abs((z - want) / want), 1) * 2.0 ** 53
    assert len(w) > 20
    assert units[~near].max() <= 3.0 + 1.0
    if near.any():
        assert units[near].max() <= 6.5 + 1.0


@pytest.mark.parametrize("which", ["radius_next_to_0", "largest_radii", "table_steps", "near_quarter_turns", "any"])
def test_normals_to_their_last_bits(blocks, which):
    w, z = blocks
    a, b = w[:, 0], w[:, 1]
    if which == "radius_next_to_0":
        pick = a >= 2 ** 32 - 2 ** 17
    elif which == "largest_radii":
        pick = a < 2 ** 17
    elif which == "table_steps":  # words of [1/2, 1) just above and below a step of 2^-9
        low = a & np.uint64(2 ** 23 - 1)
        pick = (a >= 2 ** 31) & ((low < 2 ** 10) | (low >= 2 ** 23 - 2 ** 10))
    elif which == "near_quarter_turns":
        low = b & np.uint64(2 ** 30 - 1)
        pick = np.minimum(low, 2 ** 30 - 1 - low) < 2 ** 16
    else:
        pick = np.arange(len(w)) % 40 == 0
    _check(w[pick], z[pick])
