"""The lean steps where every CTA takes several tiles (stage refill, tiles at a stride and from the counter),
bit for bit against the kernels that load per thread.  Every call runs twice on its plan: a counter left
other than zero, or a stage refilled early, shows in the second."""
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


def _problem(nx, nz, ns, nt):
    p = W.tiny(nx=nx, nz=nz, ns=ns, nt=nt, npml=5)
    p.acq.wavelet = np.repeat(p.acq.wavelet[:1], ns, 0)   # no delay from shot to shot: all have waves
    return rounded(p)


def _run(efwi, monkeypatch, p, layout, **kw):
    if layout:
        monkeypatch.setenv("EFWI_TMA_VEC", str(layout))
        monkeypatch.setenv("EFWI_ADJ_VEC", str(layout))
    plan = efwi.Plan(p.acq, exec="batched", stencil="tma_pairs" if layout else "loads", tile=(32, 16),
                     adj_stencil="tma" if layout else "loads", adj_tile=(32, 16), overlap="off", **kw)
    info = plan.info()
    assert not layout or info["layout"] == info["adj_layout"] == layout
    m = (dev(p.vp), dev(p.vs), dev(p.rho))
    d_obs = dev(W.seeded_data((p.acq.ntr, p.acq.nt), 3, 1e-9))
    out = []
    for _ in range(2):
        out += [plan.forward(*m), *plan.gradient(*m, d_obs), *plan.pseudo_hessian(*m, eps=0.02)]
        plan.sync_status()
    plan.close()
    return out


# tiles of 32 x 16 over NX = nx + 12, NZ = nz + 12: 22 x 11 x 8 = 1936 (4.2 a CTA of the forward step, 6.4 of
# the adjoint) with ragged last columns and rows; 3 x 4 x 120 = 1440 small shots, edge tiles all; 21 x 9 x 8
# = 1512, full last columns
@pytest.mark.parametrize("snap,ckpt", [("fp32", 0), ("fp16", 1000), ("bf16", 0)])
@pytest.mark.parametrize("nx,nz,ns,nt", [(673, 153, 8, 160), (84, 40, 120, 60), (660, 121, 8, 160)])
def test_several_tiles_per_cta(efwi, monkeypatch, nx, nz, ns, nt, snap, ckpt):
    p = _problem(nx, nz, ns, nt)
    kw = dict(snap_store=snap, ckpt_interval=ckpt)
    ref = _run(efwi, monkeypatch, p, 0, **kw)
    half = len(ref) // 2
    assert all(t.abs().max() > 0 for t in ref)
    for layout in (4, 5):
        out = _run(efwi, monkeypatch, p, layout, **kw)
        for k, (a, b) in enumerate(zip(out, ref)):
            assert torch.equal(a, b), (layout, k % half, k // half)
