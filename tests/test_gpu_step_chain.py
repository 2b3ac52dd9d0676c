"""Chained time steps (dependent launches; the field solve zeroes the charge for the next push)
against the same steps one call at a time, bit for bit: grids of one block and of a cluster,
bounded grids, both electron models, and two contexts interleaved on two streams."""
import pytest
import torch

import paper_1610_01071_gb300 as pe

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _ctx(ncell, ppc, stream, boundary="periodic", electrons="boltzmann", **kw):
    kin = electrons == "kinetic"
    dt = 0.005 if kin else 0.1
    c = pe.make_config(ncell, max(8, ncell // 16), 6, ncell * ppc, (0.28 if kin else 0.5) * ncell, dt, 24 * dt,
                       v_th=0.3 if kin else 1.0, seed=7, newton_tol=1e-10, newton_maxit=80, boundary=boundary,
                       electrons=electrons, sort_every=5, **kw)
    ctx = pe.Context(c, device=DEV, stream=stream)
    ctx.load_initial(profile="slab") if boundary == "absorbing" else ctx.load_initial(0.3)
    return ctx


def _state(ctx):
    ctx.stream.synchronize()
    out = [ctx.view("rho", torch.int64, ctx.cfg.ncell), ctx.view("E", torch.float64), ctx.measure()]
    for species in ["ions"] + (["electrons"] if ctx.cfg.electrons else []):
        # the counting sort does not fix the order inside a cell: compare sorted columns
        c, t, v, w = ctx.particles(species=species)
        out += [c.sort().values, (c.double() + t.double()).sort().values, v.sort().values, w.sort().values]
    torch.cuda.synchronize()
    return [x.clone() for x in out]


@pytest.mark.parametrize("ncell,ppc,kw", [(64, 33, {}), (2048, 100, {}), (8192, 256, {}),
                                          (512, 64, dict(boundary="absorbing")), (256, 70, dict(electrons="kinetic")),
                                          (128, 64, dict(electrons="kinetic", te_active=True))])
def test_chained_steps_equal_single_steps(ncell, ppc, kw):
    s1, s2 = torch.cuda.Stream(DEV), torch.cuda.Stream(DEV)
    a, b = _ctx(ncell, ppc, s1, **kw), _ctx(ncell, ppc, s2, **kw)
    torch.cuda.synchronize()
    q0 = int(a.view("rho", torch.int64, ncell).sum())
    a.pic_steps(11)
    for _ in range(11):
        b.pic_steps(1)
        s2.synchronize()
    sa, sb = _state(a), _state(b)
    for x, y in zip(sa, sb):
        assert torch.equal(x, y)
    if kw.get("boundary") != "absorbing":  # the charge grid holds the deposit of the current particles
        assert int(sa[0].sum()) == q0
    assert a.sync_status() == 0 and b.sync_status() == 0


@pytest.mark.parametrize("kw", [{}, dict(coarse="phase_space", n_v=32), dict(wavelet="d4")])
def test_bursts_on_two_streams_equal_a_lone_burst(kw):
    s1, s2 = torch.cuda.Stream(DEV), torch.cuda.Stream(DEV)
    a, b = _ctx(512, 128, s1, **kw), _ctx(512, 128, s2, **kw)
    torch.cuda.synchronize()
    lone = _ctx(512, 128, torch.cuda.Stream(DEV), **kw)
    for _ in range(3):
        lone.step()
        lone.stream.synchronize()
    for _ in range(3):
        a.step()
        b.step()
    torch.cuda.synchronize()
    for x in (a, b):
        assert torch.equal(x.get_coarse(), lone.get_coarse()) and torch.equal(x.get_slope(), lone.get_slope())
        assert x.sync_status() == 0
