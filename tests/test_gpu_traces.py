"""The adjoint source's running sums: trace and step counts below, at and past a warp's 32."""
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
