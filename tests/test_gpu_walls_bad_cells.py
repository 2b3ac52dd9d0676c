"""Plain pushes between absorbing walls with cells outside the grid: such a particle is flagged and left
as it is in memory, its weight too where another particle of its 16-byte group is absorbed in the
same step. Particles are independent, so every comparison is exact."""
import numpy as np
import pytest
import torch

import oracle as orc
import paper_1610_01071_gb300 as pe
from paper_1610_01071_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _dev(*a):
    return [torch.from_numpy(np.ascontiguousarray(x)).to(DEV) for x in a]


@pytest.mark.parametrize("ncell,N,bad", [(8, 4, [2]), (64, 131, [0, 5, 6, 64, 130]), (2048, 4097, list(range(1, 4097, 37)))])
def test_a_bad_cell_keeps_its_weight_beside_an_absorption(ncell, N, bad):
    c, t, v, w = inputs.random_particles(N, ncell - 1, seed=N)
    w = (0.5 + w).astype(np.float32)
    v *= np.float32(0.2)
    for i in bad:  # the next particle of the group leaves through the left wall
        j = (i & ~3) | ((i + 1) & 3)
        if j < N and j not in bad:
            c[j], t[j], v[j] = 0, 0.25, -4.0
    cb = c.copy()
    cb[bad] = np.resize(np.array([-1, ncell, 2**31 - 1, -(2**31), ncell + 3], np.int32), len(bad))
    keep = np.ones(N, bool)
    keep[bad] = False
    Ef = _dev(np.zeros(ncell, np.float32))[0]
    s_w = orc.fx_shift(2.0 * N)
    got, want = _dev(cb, t, v, w), _dev(c[keep], t[keep], v[keep], w[keep])
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    rho = pe.push(*got, Ef, ncell, 1.0, 0.1, 1.0, s_w, boundary="absorbing", status=st)
    assert torch.equal(rho, pe.push(*want, Ef, ncell, 1.0, 0.1, 1.0, s_w, boundary="absorbing"))
    assert int(st.item()) == 4  # range
    assert int((want[3] == 0).sum()) > 0  # particles were absorbed
    k = torch.from_numpy(keep).to(DEV)
    for a, b, orig in zip(got, want, (cb, t, v, w)):
        assert torch.equal(a[k], b)
        assert np.array_equal(a[~k].cpu().numpy(), orig[~keep])
