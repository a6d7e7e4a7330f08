"""The tile counters of the lean steps after a launch that gave up its bounded wait: no later call
depends on where it left them, and a wait that runs out while variants are timed is not forgotten."""
import ctypes as C

import numpy as np
import pytest
import torch

import workloads as W
from common import rounded

pytestmark = pytest.mark.gpu
ERR_TIMEOUT = -5


@pytest.fixture(scope="module")
def efwi():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_14130_gb300 as m
    return m


def dev(a):
    return torch.tensor(np.ascontiguousarray(np.asarray(a, np.float32)), device="cuda")


def test_calls_start_from_zero_counters(efwi, monkeypatch):
    monkeypatch.setenv("EFWI_TMA_VEC", "4")
    monkeypatch.setenv("EFWI_ADJ_VEC", "4")
    # 96 x 52 padded cells: 12 tiles a shot, three a CTA of the forward step and five of the adjoint
    # (W.tiny delays each shot's wavelet more than the one before: here all start together)
    p = W.tiny(nx=84, nz=40, ns=120, nt=60, npml=5)
    p.acq.wavelet = np.repeat(p.acq.wavelet[:1], p.acq.ns, 0)
    p = rounded(p)
    plan = efwi.Plan(p.acq, exec="batched", stencil="tma_pairs", tile=(32, 16), adj_stencil="tma",
                     adj_tile=(32, 16), overlap="off")
    info = plan.info()
    assert info["layout"] == info["adj_layout"] == 4
    m = [dev(v) for v in (p.vp, p.vs, p.rho)]
    d_obs = dev(W.seeded_data((p.acq.ntr, p.acq.nt), 3, 1e-9))

    def calls():
        return [plan.forward(*m).clone(), *plan.gradient(*m, d_obs), *plan.pseudo_hessian(*m, eps=0.02)]

    ref = calls()
    plan.sync_status()
    # every shot's data has arrived waves, so a tile left out anywhere shows
    assert (ref[0].view(p.acq.ns, -1).abs().amax(1) > 0).all()
    lib = efwi.load_library()
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    for k in range(3):                      # each of the three calls is once the first after it
        assert lib.efwi_selftest_timeout(plan._h, 1 << 21, stream) == 0
        with pytest.raises(efwi.EfwiError):
            plan.sync_status()
        out = [lambda: [plan.forward(*m)], lambda: plan.gradient(*m, d_obs),
               lambda: plan.pseudo_hessian(*m, eps=0.02)][k]()
        want = [ref[:1], ref[1:5], ref[5:]][k]
        plan.sync_status()
        assert all(torch.equal(a, b) for a, b in zip(out, want)), k
    plan.close()


def test_wait_that_expires_while_variants_are_timed_fails_the_plan(efwi, monkeypatch):
    p = rounded(W.tiny(nx=40, nz=30, ns=2, nt=20, npml=5))
    monkeypatch.setenv("EFWI_TEST_TUNE_TIMEOUT", "1")
    with pytest.raises(efwi.EfwiError) as e:
        efwi.Plan(p.acq, exec="batched")
    assert e.value.code == ERR_TIMEOUT and "bounded wait" in str(e.value)
    monkeypatch.delenv("EFWI_TEST_TUNE_TIMEOUT")
    plan = efwi.Plan(p.acq, exec="batched")
    plan.forward(*[dev(v) for v in (p.vp, p.vs, p.rho)])
    plan.sync_status()
    plan.close()
