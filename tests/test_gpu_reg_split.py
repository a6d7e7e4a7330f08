"""Consistency term and collapse at the ends of every split of a pixel's components over threads, and
where the sums need care: sinkholes on the first or on all components, values that one FP32 sum does not
hold.  Reference: the FP64 oracle."""
import ctypes as C

import numpy as np
import pytest
import torch

import workloads as W
from common import f32, rel_l2
from oracle import extension as X

pytestmark = pytest.mark.gpu
NZ, NX = 19, 41                                           # 779 pixels: ragged blocks of 32 to 256


@pytest.fixture(scope="module")
def efwi():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_14130_gb300 as m
    return m


def dev(a, dtype=np.float32):
    return torch.tensor(np.ascontiguousarray(np.asarray(a, dtype)), device="cuda")


def _weights(ns, seed, sinks=0.3):
    rng = np.random.default_rng(seed)
    b = f32(rng.uniform(0.05, 1.0, (ns, NZ, NX)))
    sink = (rng.random((ns, NZ, NX)) < sinks / ns).astype(np.uint8)
    sink[:, :7] = 0                                       # rows of pixels without any
    return rng, b, np.where(sink, 1.0, b), sink


def _check(efwi, m, b, bp, sink, tol_phi, tol_g=1e-6):
    """phi, gradient (both entry points) and collapse against the oracle."""
    plan = efwi.Plan(W.tiny(nx=NX, nz=NZ, ns=2, nt=4, npml=3).acq, exec="plain")
    args = dev(m), dev(b), dev(bp), dev(sink, np.uint8)
    phi_o, g_o = X.regularization(m, b, bp, sink, 0.7)
    phi, g = plan.regularization_grad(*args, 0.7)
    phi2, g2 = torch.empty((), dtype=torch.float64, device="cuda"), torch.zeros_like(g)
    ptr = [C.c_void_p(t.data_ptr()) for t in (*args, phi2, g2)]
    assert efwi.load_library().efwi_regularization_grad_noalloc(
        len(m), NX, NZ, *ptr[:4], 0.7, *ptr[4:], C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    plan.close()
    assert torch.equal(g, g2)
    for v in (phi, phi2):
        assert abs(v.item() - phi_o) <= tol_phi * phi_o
    assert rel_l2(g.cpu().numpy(), g_o) <= tol_g
    out = efwi.collapse(*args).cpu().numpy()
    assert rel_l2(out, X.collapse(m, b, bp, sink)) <= 1e-6


# phi: pairs of FP32 (2^-47) amplified by at most 2 ns, and the oracle's own FP64 sums
@pytest.mark.parametrize("kind", ["near", "spread", "signed"])
@pytest.mark.parametrize("ns", [2, 3, 4, 5, 8, 9, 16, 17, 32, 33, 64, 65, 128, 129, 256, 257])
def test_ends_of_the_splits(efwi, ns, kind):
    rng, b, bp, sink = _weights(ns, 100 + ns)
    z = rng.standard_normal((ns, NZ, NX))
    m = {"near": 3000 + 100 * z, "spread": 10.0 ** (2 * z), "signed": 1e-9 * z * np.exp(2 * z[::-1])}[kind]
    _check(efwi, f32(m), b, bp, sink, 1e-10)


def test_one_component(efwi):
    # the residual is zero, with or without a sinkhole
    _, b, bp, sink = _weights(1, 3)
    m = f32(np.random.default_rng(3).uniform(1500, 4000, (1, NZ, NX)))
    plan = efwi.Plan(W.tiny(nx=NX, nz=NZ, ns=2, nt=4, npml=3).acq, exec="plain")
    phi, g = plan.regularization_grad(dev(m), dev(b), dev(bp), dev(sink, np.uint8), 0.7)
    assert phi.item() == 0.0 and float(g.abs().max()) == 0.0
    assert np.array_equal(efwi.collapse(dev(m), dev(b), dev(bp), dev(sink, np.uint8)).cpu().numpy(), np.float32(m[0]))
    plan.close()


# the first component, or every one, has its sinkhole at a pixel and is far (D = 1000) from the others,
# whose residual is r = 0.05: a pivot there would cost (D / r)^2 = 4e8 of the sums' 47 or 53 bits.  The
# oracle's residuals carry 2^-53 of 3000, 7e-12 of r.
# (Two components alone would take each other's value there.)
@pytest.mark.parametrize("ns,sinks", [(n, k) for n in (2, 4, 8, 16, 64, 257) for k in ("first", "all") if n > 2 or k == "first"])
def test_sinkhole_of_the_first_component(efwi, ns, sinks):
    rng = np.random.default_rng(ns)
    m = 3000 + 0.05 * rng.standard_normal((ns, NZ, NX))
    b = rng.uniform(0.3, 1.0, (ns, NZ, NX))
    m[0], b[0] = 4000.0, 1e-7
    sink = np.zeros((ns, NZ, NX), np.uint8)
    sink[0, :, ::2] = 1
    if sinks == "all":
        sink[:, :, ::2] = 1
    b = f32(b)
    m, bp = f32(m), np.where(sink, 0.5, b)
    m[0, :, 1::2] = f32(3000.0)                           # no outlier where it has no sinkhole
    _check(efwi, m, b, bp, sink, 1e-9)


# weights whose FP32 sum overflows; a component of weight 0 that is larger than all digits of the rest
@pytest.mark.parametrize("ns", [2, 4, 7, 20])
def test_collapse_of_extreme_weights_and_values(efwi, ns):
    rng, b, bp, sink = _weights(ns, 7, sinks=0.0)
    m = f32(rng.uniform(1500, 4000, (ns, NZ, NX)))
    out = efwi.collapse(dev(m), dev(b), dev(bp * 3e38), dev(sink, np.uint8)).cpu().numpy()
    assert rel_l2(out, X.collapse(m, b, np.float32(bp * 3e38).astype(np.float64), sink)) <= 1e-6
    if ns > 2:
        m[0], bp[0] = 1e30, 0.0
        out = efwi.collapse(dev(m), dev(b), dev(bp), dev(sink, np.uint8)).cpu().numpy()
        assert rel_l2(out, X.collapse(m, b, bp, sink)) <= 1e-6


@pytest.mark.parametrize("ns", [2, 4, 7, 20])
@pytest.mark.parametrize("s", [0, 1])
def test_collapse_of_an_infinity(efwi, ns, s):
    _, b, bp, sink = _weights(ns, 9, sinks=0.0)
    m = np.full((ns, NZ, NX), 2000.0)
    m[s, 4, 40], m[s, 11, 3] = np.inf, -np.inf
    out = efwi.collapse(dev(m), dev(b), dev(bp), dev(sink, np.uint8)).cpu().numpy()
    assert out[4, 40] == np.inf and out[11, 3] == -np.inf
    assert np.isfinite(out).sum() == NZ * NX - 2
