"""DAS sampling inside the forward step and the adjoint source's running sums: trace counts below, at
and past a warp's 32 and a CTA's 256, on CTAs of their own and, where the tiles fill the device, on
CTAs that also have tiles."""
import numpy as np
import pytest
import torch

import workloads as W
from common import f32, rel_l2, rounded
from oracle import elastic as E

pytestmark = pytest.mark.gpu
TOL = 1e-4      # FP32 time stepping against the FP64 oracle, as for every data and gradient comparison


@pytest.fixture(scope="module")
def efwi():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_14130_gb300 as m
    return m


def dev(a):
    return torch.tensor(np.ascontiguousarray(np.asarray(a, np.float32)), device="cuda")


# 672 x 42 padded cells: 63 tiles a shot, 504 for eight, more than the 456 CTAs resident at once
@pytest.mark.parametrize("nx,nz,ns,nch,mode", [(40, 30, 2, 6, W.STRAIN), (40, 30, 1, 256, W.STRAIN_RATE),
                                               (41, 33, 1, 257, W.STRAIN), (660, 30, 8, 5, W.STRAIN),
                                               (660, 30, 8, 40, W.STRAIN)])
def test_step_samples_the_traces_of_the_step_before(efwi, monkeypatch, nx, nz, ns, nch, mode):
    p = rounded(W.tiny(nx=nx, nz=nz, ns=ns, nt=41, npml=5, das_mode=mode, nch=nch))
    m = (dev(p.vp), dev(p.vs), dev(p.rho))
    out = []
    for layout in (0, 4, 5):
        if layout:
            monkeypatch.setenv("EFWI_TMA_VEC", str(layout))
        plan = efwi.Plan(p.acq, exec="batched" if layout else "plain", stencil="tma_pairs" if layout else "auto",
                         tile=(32, 16))
        assert not layout or plan.info()["layout"] == layout
        out += [plan.forward(*m), plan.forward(*m)]
        plan.close()
    assert out[0].abs().max() > 0
    for d in out[1:]:
        assert torch.equal(d, out[0])


@pytest.mark.parametrize("nt", [1, 31, 32, 33, 65])
@pytest.mark.parametrize("ns,nch", [(1, 1), (1, 32), (2, 33)])
@pytest.mark.parametrize("exec_", ["plain", "batched"])
def test_adjoint_source_of_strain_data(efwi, nt, ns, nch, exec_):
    p = rounded(W.tiny(nx=36, nz=28, ns=ns, nt=nt, npml=4, nch=nch))
    # data far from the modelled ones, so that the residual is not zero before the waves arrive
    d_obs = f32(W.seeded_data((p.acq.ntr, p.acq.nt), 5, 1e-9))
    phi_o, *g_o = E.gradient(p.acq, p.vp, p.vs, p.rho, d_obs)
    plan = efwi.Plan(p.acq, exec=exec_)
    phi, *g = plan.gradient(dev(p.vp), dev(p.vs), dev(p.rho), dev(d_obs))
    torch.cuda.synchronize()
    assert abs(phi.item() - phi_o) <= TOL * phi_o
    for a, b in zip(g, g_o):
        assert rel_l2(a.cpu().numpy(), b) <= TOL
    plan.close()
