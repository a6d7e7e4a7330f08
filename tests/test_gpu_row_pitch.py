"""Plans whose rows fall back to multiples of 8 cells because the workspace does not fit with rows of 32:
the same bits from every call, in less memory."""
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


# NX + 8 = nx + 20: rows of 72 for 96, of 8 more than a tile column, and windows of four widths
@pytest.mark.parametrize("snap", ["fp32", "fp16"])
@pytest.mark.parametrize("nx,win", [(45, None), (53, None), (170, [[20, 90], [13, 157], [60, 50], [0, 170]])])
@pytest.mark.parametrize("layout", [0, 1, 3, 4, 5])
def test_short_rows_give_the_same_bits(efwi, monkeypatch, nx, win, snap, layout):
    p = rounded(W.tiny(nx=nx, nz=33, ns=4, nt=40, npml=5, win=win))
    m = (dev(p.vp), dev(p.vs), dev(p.rho))
    d_obs = dev(W.seeded_data((p.acq.ntr, p.acq.nt), 3, 1e-9))
    if layout:
        monkeypatch.setenv("EFWI_TMA_VEC", str(layout))
        monkeypatch.setenv("EFWI_ADJ_VEC", str(layout))
    out, size = [], []
    for fail in ("0", "-3"):
        monkeypatch.setenv("EFWI_TEST_FAIL_ALLOC", fail)
        plan = efwi.Plan(p.acq, exec="batched", stencil=("loads", "tma")[layout == 1] if layout < 2 else "tma_pairs",
                         tile=(32, 16), adj_stencil="tma" if layout else "loads", adj_tile=(32, 16), overlap="off",
                         snap_store=snap)
        out.append([plan.forward(*m), *plan.gradient(*m, d_obs), *plan.pseudo_hessian(*m, eps=0.02)])
        plan.sync_status()
        size.append(plan.info()["workspace_bytes"])
        plan.close()
    assert size[1] < size[0]
    assert all(t.abs().max() > 0 for t in out[0])
    assert all(torch.equal(a, b) for a, b in zip(*out))
