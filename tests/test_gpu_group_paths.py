"""Particle passes on groups that leave the usual window: few particles per cell, velocities in no
order, and cells outside the grid at any place of a 16-byte group, a warp or the ragged tail. All
sums are integers, so every comparison is exact."""
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


def _sample(kind, ncell, s_w, E0):
    nb = ncell >> 2
    if kind == "none":
        return None, None
    rows = torch.zeros((nb, 16) if kind == "phase" else (2, nb), dtype=torch.int64, device=DEV)
    kw = dict(n_v=16, v_min=-8.0, dv=1.0) if kind == "phase" else {}
    return rows, pe.make_sample_args(E0, 3.0, 1.0, 2.0, s_w, s_w - 5, rows, bin_shift=2, **kw)


@pytest.mark.parametrize("kind", ["none", "moments", "phase"])
@pytest.mark.parametrize("ncell,N,bad", [(8, 3, [1]), (64, 131, [0, 5, 6, 7, 130]), (1024, 40001, [0, 127, 128, 4095, 40000]),
                                         (4096, 9000, list(range(64, 96)))])
def test_cells_outside_the_grid_are_left_alone(ncell, N, bad, kind):
    c, t, v, w = inputs.random_particles(N, ncell, seed=N)
    v *= np.float32(4.0)  # a group's new cells spread over many
    s_w = orc.fx_shift(2.0 * ncell / N)
    cb = c.copy()
    cb[bad] = np.resize(np.array([-1, ncell, 2**31 - 1, -(2**31), ncell + 3], np.int32), len(bad))
    keep = np.ones(N, bool)
    keep[bad] = False
    Ef = inputs.random_field(ncell, 3).astype(np.float32)
    got, want = _dev(cb, t, v, w), _dev(c[keep], t[keep], v[keep], w[keep])
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    E0 = torch.zeros(ncell, device=DEV)
    rows, args = _sample(kind, ncell, s_w, E0)
    rows2, args2 = _sample(kind, ncell, s_w, E0)
    # the deposit and the sample before the push, then the push
    assert torch.equal(pe.deposit(got[0], got[1], got[3], ncell, s_w, status=st), pe.deposit(want[0], want[1], want[3], ncell, s_w))
    if args is not None:
        pe.sample(*got, _dev(Ef)[0], ncell, 0.1, 1.0, args, status=st)
        pe.sample(*want, _dev(Ef)[0], ncell, 0.1, 1.0, args2)
        assert torch.equal(rows, rows2)
    assert int(st.item()) == 4  # range
    st.zero_()
    rho = pe.push(*got, _dev(Ef)[0], ncell, 0.7, 0.1, 1.0, s_w, sample=args, status=st)
    assert torch.equal(rho, pe.push(*want, _dev(Ef)[0], ncell, 0.7, 0.1, 1.0, s_w, sample=args2))
    assert int(st.item()) == 4
    if args is not None:
        assert torch.equal(rows, rows2)
    k = torch.from_numpy(keep).to(DEV)
    for a, b, orig in zip(got, want, (cb, t, v, w)):
        assert torch.equal(a[k], b)
        assert np.array_equal(a[~k].cpu().numpy(), orig[~keep])


@pytest.mark.parametrize("ncell,ppc,spread", [(256, 1, 0.5), (2048, 3, 3.0), (128, 900, 0.3), (128, 900, 2.0), (1024, 40, 30.0)])
def test_unordered_groups_deposit_exactly(ncell, ppc, spread):
    N = ncell * ppc + 5
    c, t, v, w = inputs.random_particles(N, ncell, seed=ppc)
    s_w = orc.fx_shift(2.0 * ncell / N)
    for kind in ("none", "moments"):
        E0 = torch.zeros(ncell, device=DEV)
        rows, args = _sample(kind, ncell, s_w, E0)
        d = _dev(c, t, v * np.float32(spread), w)
        for _ in range(3):
            rho = pe.push(*d, torch.zeros(ncell, device=DEV), ncell, 1.0, 0.1, 1.0, s_w, sample=args)
            gc, gt, _, gw = [x.cpu().numpy() for x in d]
            assert np.array_equal(rho.cpu().numpy(), orc.deposit_fx(gc, gt, gw, ncell, s_w))
