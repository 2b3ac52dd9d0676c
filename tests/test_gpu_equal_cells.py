"""Equal-weight loading where a thread block's points span few or many cells: the cells staged in
shared memory (at most 512 of a block), the global table beyond that (a near vacuum), the ragged tail
and the smallest grid, against the FP64 CPU oracle.

Positions agree within 2e-6 cell per 1024 nodes (FP32 offsets; the cell of a point on an edge may differ,
its position not), weights within 1e-7 relative, velocities within 2e-5; the deposit is that of
pe_deposit on the loaded particles, bit for bit."""
import numpy as np
import pytest
import torch

import oracle as orc
import paper_1610_01071_gb300 as pe
from paper_1610_01071_gb300 import _binding as pb

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def profile(n, thin):
    """Uniform, or falling to a thin floor that most of the grid holds (smoothly: a cell's density keeps
    the FP32 offset well conditioned)."""
    j = np.arange(n)
    return np.maximum(np.exp(-j / max(n / 64, 2.0)), 1e-3) if thin else np.ones(n)


@pytest.mark.parametrize("thin", [False, True])
@pytest.mark.parametrize("ncell,N", [(8, 5), (8, 4097), (512, (1 << 15) + 1), (1024, 1 << 18), (8192, 1 << 18),
                                     (8192, 12289)])
def test_moment_loader(ncell, N, thin):
    n = profile(ncell, thin).astype(np.float32)
    u = (0.2 * np.sin(2 * np.pi * np.arange(ncell) / ncell)).astype(np.float32)
    s_w = orc.fx_shift(4.0 * ncell / N)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    cell, theta, v, w, rho = pe.quiet_start_equal(N, ncell, torch.from_numpy(n).to(DEV), torch.from_numpy(u).to(DEV),
                                                  1.0, 7, s_w, status=st)
    so = orc.quiet_start_equal(N, ncell, n.astype(np.float64), u.astype(np.float64), 1.0, 7)
    assert int(st.item()) == 0
    x = cell.cpu().numpy() + theta.cpu().numpy().astype(np.float64)
    assert np.max(np.abs(x - (so.cell + so.theta))) < 2e-6 * max(1.0, ncell / 1024)
    assert np.allclose(w.cpu().numpy(), so.w, rtol=1e-7)
    assert np.max(np.abs(v.cpu().numpy() - so.v)) < 2e-5
    assert torch.equal(rho, pe.deposit(cell, theta, w, ncell, s_w))


@pytest.mark.parametrize("thin", [False, True])
@pytest.mark.parametrize("ncell,b,N", [(8, 0, 5), (256, 3, 4097), (1024, 4, 1 << 18), (8192, 5, (1 << 18) + 2)])
def test_phase_space_loader(ncell, b, N, thin):
    nxc, nv = ncell >> b, 16
    vmin, dv = -6.0, 12.0 / nv
    vc = vmin + dv * (np.arange(nv) + 0.5)
    H = profile(nxc, thin)[:, None] * (1 << b) * np.exp(-0.5 * vc[None, :] ** 2) * dv
    mass, cdf, table, _ = pb.ps_lift_tables(torch.from_numpy(H).to(DEV))
    s_w = orc.fx_shift(4.0 * float(mass.sum()) / N)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    cell, theta, v, w, rho = pb.ps_quiet_start_equal(N, ncell, b, mass, table, vmin, dv, 3, s_w, status=st)
    so = orc.ps_quiet_start_equal(N, ncell, b, mass.cpu().numpy(), cdf.cpu().numpy(), vmin, dv, 3)
    assert int(st.item()) == 0
    x = cell.cpu().numpy() + theta.cpu().numpy().astype(np.float64)
    assert np.max(np.abs(x - (so.cell + so.theta))) < 2e-6 * max(1.0, ncell / 1024)
    assert np.allclose(w.cpu().numpy(), so.w, rtol=1e-7)
    dv_ = np.abs(v.cpu().numpy() - so.v)  # a cell whose density vanishes at an edge: see test_gpu_walls
    assert dv_.max() <= 0.2 * dv and np.sum(dv_ > 5e-5) <= max(3, 1e-4 * N)
    assert torch.equal(rho, pe.deposit(cell, theta, w, ncell, s_w))
