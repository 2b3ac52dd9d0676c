"""Lifting profiles and projections where their blocks' shares end: grids smaller than the number of
blocks, densities with and without negative values (clamped, total kept), bursts of more pairs of samples
than a block stages at once, component counts off the block size. FP64 against the CPU oracle: the same
sums in another order, 1e-12 of the largest value; profiles are FP32, one rounding (6e-8 relative)."""
import numpy as np
import pytest
import torch

import oracle as orc
import paper_1610_01071_gb300 as pe

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("negative", [False, True])
@pytest.mark.parametrize("ncell,nc,wav", [(4, 4, "haar"), (8, 2, "haar"), (64, 64, "haar"), (256, 32, "coif4"),
                                          (4096, 64, "haar"), (8192, 256, "coif4")])
def test_refine_profiles(ncell, nc, wav, negative):
    rng = np.random.default_rng(ncell + nc + negative)
    c = np.stack([1.0 + 0.1 * rng.random(nc), 0.3 * rng.standard_normal(nc)])
    if negative:
        c[0, nc // 2] = -0.4
    pn, pu = pe.refine(torch.from_numpy(c).to(DEV), ncell, wavelet=wav)
    n, u = orc.lift_profile(orc.refine(c[0], ncell, wav), orc.refine(c[1], ncell, wav))
    assert np.allclose(pn.cpu().numpy(), n, rtol=2e-7, atol=1e-12 * np.abs(n).max())
    big = n > 1e-6 * n.max()  # the velocity is set to 0 at the density's floor
    assert np.allclose(pu.cpu().numpy()[big], u[big], rtol=2e-7, atol=1e-9 * np.abs(u).max())


@pytest.mark.parametrize("K", [2, 3, 20, 127, 128, 300])
@pytest.mark.parametrize("ncoef", [1, 63, 65, 512])
def test_ls_project(K, ncoef):
    rng = np.random.default_rng(K + ncoef)
    y = rng.standard_normal((K + 1, ncoef))
    out, slope = pe.ls_project(torch.from_numpy(y).to(DEV), 0.1, 20.0 + 0.1 * K)
    want, wslope = orc.ls_project(y, 0.1, 20.0 + 0.1 * K)
    assert np.allclose(slope.cpu().numpy(), wslope, rtol=0, atol=1e-12 * (1.0 + np.abs(wslope).max()))
    assert np.allclose(out.cpu().numpy(), want, rtol=0, atol=1e-12 * (1.0 + np.abs(want).max()))
