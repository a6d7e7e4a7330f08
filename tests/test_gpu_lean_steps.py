"""The lean forward and adjoint steps (EFWI_TMA_VEC, EFWI_ADJ_VEC = 4 and 5) against the kernels that
load per thread, bit for bit: grids that end inside, at and just past a 32 x 16 tile (odd and even widths),
windows, force sources, every snapshot store."""
import numpy as np
import pytest
import torch

import workloads as W
from common import rounded

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def efwi():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_14130_gb300 as m
    return m


def dev(a):
    return torch.tensor(np.ascontiguousarray(np.asarray(a, np.float32)), device="cuda")


def _run(efwi, monkeypatch, p, layout, **kw):
    if layout:
        monkeypatch.setenv("EFWI_TMA_VEC", str(layout))
        monkeypatch.setenv("EFWI_ADJ_VEC", str(layout))
    # the reference shares no copy with the lean steps: its threads load cell by cell
    plan = efwi.Plan(p.acq, exec="batched", stencil="tma_pairs" if layout else "loads", tile=(32, 16),
                     adj_stencil="tma" if layout else "loads", adj_tile=(32, 16), overlap="off", **kw)
    info = plan.info()
    assert not layout or info["layout"] == info["adj_layout"] == layout
    m = (dev(p.vp), dev(p.vs), dev(p.rho))
    d_obs = dev(W.seeded_data((p.acq.ntr, p.acq.nt), 3, 1e-9))
    # forward data, misfit, gradients and the gradient call's own data
    out = [plan.forward(*m)] + list(plan.gradient(*m, d_obs, return_data=True))
    plan.sync_status()
    plan.close()
    return out


# NX = nx + 12, NZ = nz + 12: one column or row past a tile, one short of it, exact, in between
@pytest.mark.parametrize("nx,nz", [(40, 30), (52, 36), (51, 35), (53, 37), (84, 53), (115, 21), (20, 17)])
def test_lean_step_equals_single_cells(efwi, monkeypatch, nx, nz):
    p = rounded(W.tiny(nx=nx, nz=nz, ns=2, nt=36, npml=5))
    ref = _run(efwi, monkeypatch, p, 0)
    for layout in (4, 5):
        for a, b in zip(_run(efwi, monkeypatch, p, layout), ref):
            assert torch.equal(a, b), layout


@pytest.mark.parametrize("source", ["moment_tensor", "force"])
@pytest.mark.parametrize("snap", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("ckpt", [0, 1000])
def test_lean_step_windows_sources_and_snapshots(efwi, monkeypatch, source, snap, ckpt):
    p = rounded(W.tiny(nx=170, nz=45, ns=4, nt=40, npml=5, win=[[20, 90], [13, 157], [60, 50], [0, 170]]))
    if source == "force":
        p = W.with_forces(p)
    kw = dict(snap_store=snap, ckpt_interval=ckpt)
    ref = _run(efwi, monkeypatch, p, 0, **kw)
    for layout in (4, 5):
        for a, b in zip(_run(efwi, monkeypatch, p, layout, **kw), ref):
            assert torch.equal(a, b), layout


# the step's own sum of |v|^2 and the pass that follows a step of the kernels that load per thread
@pytest.mark.parametrize("nx,nz,win", [(52, 36, None), (51, 35, None), (53, 37, None),
                                       (170, 45, [[20, 90], [13, 157], [0, 170]])])
def test_lean_step_sums_the_energy(efwi, monkeypatch, nx, nz, win):
    p = rounded(W.tiny(nx=nx, nz=nz, ns=3, nt=36, npml=5, win=win))
    out = []
    for layout in (0, 4, 5):
        if layout:
            monkeypatch.setenv("EFWI_TMA_VEC", str(layout))
        plan = efwi.Plan(p.acq, exec="batched", stencil="tma_pairs" if layout else "loads", tile=(32, 16))
        assert not layout or plan.info()["layout"] == layout
        out.append(plan.pseudo_hessian(dev(p.vp), dev(p.vs), dev(p.rho), eps=0.02))
        plan.sync_status()
        plan.close()
    for h, hi in out[1:]:
        assert torch.equal(h, out[0][0]) and torch.equal(hi, out[0][1])
