"""Field solves: the returned field is the centred difference of the returned potential, to the bit, at
every node. Warps and blocks difference their edge nodes against copies of the neighbours' potential
that they advance themselves, so one copy off by a rounding shows here."""
import numpy as np
import pytest
import torch

import paper_1610_01071_gb300 as pe

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
S_W = 20


def _rho(n, kind, g):
    x = torch.arange(n, dtype=torch.float64, device=DEV) / n
    noise = 1.0 + 0.05 * torch.randn(n, generator=g, dtype=torch.float64, device=DEV)
    base = torch.sigmoid((0.0625 - (x - 0.5).abs()) * 200.0) if kind == "absorbing" else 1.0 + 0.5 * torch.sin(6.2831853 * x)
    return torch.round((base * noise).clamp(min=0.0) * 2.0 ** (S_W + 24)).to(torch.int64)


@pytest.mark.parametrize("boundary", ["periodic", "absorbing"])
@pytest.mark.parametrize("n", [8, 32, 64, 256, 512, 1024, 4096, 8192])
def test_the_field_is_the_difference_of_the_potential(n, boundary):
    g = torch.Generator(device=DEV).manual_seed(n)
    for mode in ("boltzmann", "linearized"):
        for dx, phi0, maxit in ((0.5, 0.0, 200), (0.3, 0.0, 1), (0.3, -9.0, 3), (0.5, 6.0, 200), (0.37, 0.0, 0)):  # +-: damped steps
            rho = _rho(n, boundary, g)
            phi = phi0 * torch.rand(n, generator=g, dtype=torch.float64, device=DEV)
            E, Ef, _ = pe.field(rho, n, dx, S_W, phi, mode=mode, tol=1e-10, maxit=maxit, boundary=boundary)
            want = (phi.roll(1) - phi.roll(-1)) * (0.5 / dx)
            if boundary == "absorbing":
                want[0] = want[-1] = 0.0
            assert torch.equal(E, want), (mode, dx, phi0, int((E != want).sum()))
            assert torch.equal(Ef, want.float())


@pytest.mark.parametrize("n", [64, 1024])
def test_a_tolerance_below_single_precision_still_ends_an_exact_solve(n):
    rho = torch.full((n,), 1 << (S_W + 24), dtype=torch.int64, device=DEV)  # density 1: phi = 0 is exact
    phi = torch.zeros(n, dtype=torch.float64, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    E, _, diag = pe.field(rho, n, 0.5, S_W, phi, mode="linearized", tol=1e-60, maxit=9, status=st)
    assert diag.tolist()[:2] == [1, 1] and int(st.item()) == 0
    assert float(E.abs().max()) == 0.0 and float(phi.abs().max()) == 0.0


@pytest.mark.parametrize("boundary", ["periodic", "absorbing"])
@pytest.mark.parametrize("n", [8, 16])
def test_the_smallest_grids_solve_to_rounding(n, boundary):
    g = torch.Generator(device=DEV).manual_seed(n + 1)
    dx = 0.4
    for mode in ("boltzmann", "linearized"):
        for _ in range(6):
            rho = _rho(n, "periodic", g)  # no vacuum: a well-conditioned Jacobian
            phi = torch.zeros(n, dtype=torch.float64, device=DEV)
            pe.field(rho, n, dx, S_W, phi, mode=mode, tol=1e-10, maxit=50, boundary=boundary)
            d = rho.cpu().numpy() * 2.0 ** -(S_W + 24)
            if boundary == "absorbing":
                d[0] *= 2.0
                d[-1] *= 2.0
            L = (2.0 * np.eye(n) - np.roll(np.eye(n), 1, 1) - np.roll(np.eye(n), -1, 1)) / dx**2
            if boundary == "absorbing":  # mirror ghosts
                L[0], L[-1] = 0.0, 0.0
                L[0, 0] = L[-1, -1] = 2.0 / dx**2
                L[0, 1] = L[-1, -2] = -2.0 / dx**2
            p = np.zeros(n)
            for _ in range(30):
                e, de = (np.exp(p), np.exp(p)) if mode == "boltzmann" else (1.0 + p, np.ones(n))
                p = p - np.linalg.solve(L + np.diag(de), L @ p + e - d)
            # rounding: a few 2^-53 of the terms of F, at most 4 max|phi| / dx^2, over min g' (> 0.2 here)
            assert np.max(np.abs(phi.cpu().numpy() - p)) < 4e-14 * max(1.0, np.max(np.abs(p))), (mode, n)
