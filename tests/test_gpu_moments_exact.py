"""The particle moments against exact rational sums: the three-float sums are rounded once, at their
conversion to FP64; particles whose products leave FP32's range, counts that are no multiple of
four and arrays that are not 16-byte aligned take other paths to the same sums."""
from fractions import Fraction

import numpy as np
import pytest
import torch

import paper_1610_01071_gb300 as pe
from paper_1610_01071_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("N,shift,extreme", [(1, 0, False), (2003, 0, False), (2003, 1, False), (1500, 0, True),
                                             (4099, 3, True)])
def test_moments_equal_exact_sums(N, shift, extreme):
    ncell, dx = 64, 0.5
    c, t, v, w = inputs.random_particles(N, ncell, seed=N + shift)
    if extreme:  # cold, fast, weightless and heavy particles among the others
        rng = np.random.default_rng(N)
        v[rng.integers(0, N, 40)] *= np.float32(1e-30)
        v[rng.integers(0, N, 20)] = np.float32(3e18)
        v[rng.integers(0, N, 20)] = 0.0
        w[rng.integers(0, N, 20)] = 0.0
    # a leading pad of `shift` elements leaves the arrays off the 16-byte grid
    dev = [torch.from_numpy(np.concatenate([np.zeros(shift, a.dtype), a])).to(DEV)[shift:] for a in (c, t, v, w)]
    got = pe.compute_moments(*dev, torch.zeros(ncell, device=DEV), ncell, dx, 0.1, 0.1, 1.0, 10)  # E = 0: Vbar = v
    W, V = [Fraction(float(x)) for x in w], [Fraction(float(x)) for x in v]
    want = dict(charge=sum(W), momentum=sum(a * b for a, b in zip(W, V)),
                kinetic=sum(a * b * b for a, b in zip(W, V)) / 2)
    size = dict(charge=want["charge"], momentum=sum(abs(a * b) for a, b in zip(W, V)), kinetic=want["kinetic"])
    # one rounding per block sum and per product with dx (exact), FP64 throughout for the extreme ones:
    # at most a few units in the last place of the terms' size
    tol = 2.0**-53 * (4 if not extreme else 64)
    for k in want:
        assert abs(Fraction(got[k]) - want[k] * Fraction(dx)) <= Fraction(tol) * size[k] * Fraction(dx), k
    assert got["invalid"] == 0 and got["max_speed"] == float(np.max(np.abs(v)))
