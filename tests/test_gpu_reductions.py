"""Reductions formed in FP32 with their rounding errors carried along: the consistency term and
the collapse over every branch of their component split, and the l-BFGS inner products over
tails, alignments and magnitudes, against FP64."""
import numpy as np
import pytest
import torch

import workloads as W
from common import f32, rel_l2
from oracle import extension as X
from oracle import lbfgs as L

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def efwi():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_14130_gb300 as m
    return m


def dev(a, dtype=np.float32):
    return torch.tensor(np.ascontiguousarray(np.asarray(a, dtype)), device="cuda")


def _case(ns, nz, nx, seed):
    rng = np.random.default_rng(seed)
    b = f32(rng.uniform(0.05, 1.0, (ns, nz, nx)))
    sink = (rng.random((ns, nz, nx)) < 0.3 / ns).astype(np.uint8)
    sink[:, 0, :] = 0                                   # pixels without and with sinkholes in one block
    bp = np.where(sink, 1.0, b)
    return rng, b, bp, sink


# components per thread 2, 4, 8, 16, 32 and re-read (more than 256), at both ends of most; 851
# pixels leave a ragged block.  Sums err by about 2^-47 of sum |x|, of which phi cancels at most
# a factor ns; a gradient element is one FP32 expression (a few 2^-24).
@pytest.mark.parametrize("kind", ["near", "spread", "large", "small"])
@pytest.mark.parametrize("ns", [2, 8, 16, 17, 33, 64, 65, 129, 256, 257])
def test_consistency_term_and_collapse(efwi, ns, kind):
    nz, nx = 23, 37
    rng, b, bp, sink = _case(ns, nz, nx, ns)
    m = {"near": 3000 + 100 * rng.standard_normal((ns, nz, nx)),      # exact differences
         "spread": 10.0 ** rng.uniform(-3, 3, (ns, nz, nx)),          # components far apart
         "large": 1e19 * rng.standard_normal((ns, nz, nx)),           # squares leave FP32
         "small": 1e-21 * rng.standard_normal((ns, nz, nx))}[kind]
    m = f32(m)
    plan = efwi.Plan(W.tiny(nx=nx, nz=nz, ns=2, nt=4, npml=3).acq, exec="plain")
    # nz, nx of the weights are the plan's
    phi_o, g_o = X.regularization(m, b, bp, sink, 0.7)
    phi, g = plan.regularization_grad(dev(m), dev(b), dev(bp), dev(sink, np.uint8), 0.7)
    assert abs(phi.item() - phi_o) <= 1e-10 * phi_o
    assert rel_l2(g.cpu().numpy(), g_o) <= 1e-6
    out = efwi.collapse(dev(m), dev(b), dev(bp), dev(sink, np.uint8))
    assert rel_l2(out.cpu().numpy(), X.collapse(m, b, bp, sink)) <= 1e-6
    plan.close()


def test_consistency_term_keeps_non_finite_values_to_their_pixel(efwi):
    nz, nx, ns = 20, 70, 6
    _, b, bp, sink = _case(ns, nz, nx, 1)
    m = np.full((ns, nz, nx), 2000.0)
    m[3, 2, 40], m[0, 1, 7] = np.nan, np.inf
    plan = efwi.Plan(W.tiny(nx=nx, nz=nz, ns=2, nt=4, npml=3).acq, exec="plain")
    phi, g = plan.regularization_grad(dev(m), dev(b), dev(bp), dev(sink, np.uint8), 0.7)
    bad = ~np.isfinite(g.cpu().numpy())
    assert np.isnan(phi.item())
    assert bad[:, 2, 40].all() and bad[:, 1, 7].all() and bad.sum() == 2 * ns
    plan.close()


# tails of a block's 2048 elements, one element, more than one pass of the 1216-block grid; the
# caller's gradient and direction 16-byte aligned or not; magnitudes whose products leave FP32
@pytest.mark.parametrize("scale", [1.0, 1e-24, 1e16])
@pytest.mark.parametrize("n,shift", [(1, 0), (7, 1), (2047, 0), (2049, 3), (2_490_373, 1)])
def test_direction_over_tails_alignments_and_magnitudes(efwi, n, shift, scale):
    from paper_2305_14130_gb300.optim import LBFGS
    rng = np.random.default_rng(n)
    a = rng.uniform(0.5, 5.0, n)
    S = np.float32(scale * rng.standard_normal((3, n)))
    Y = np.float32(S * a)
    g = np.float32(scale * rng.standard_normal(n))
    opt = LBFGS(n, m=3)
    for s, y in zip(S, Y):
        assert opt.push(dev(s), dev(y))
    gd = torch.zeros(n + 4, device="cuda")[shift:shift + n]
    gd.copy_(dev(g))
    d = opt.direction(gd).cpu().numpy()
    ref = -L.two_loop(g.astype(np.float64), S.astype(np.float64), Y.astype(np.float64))
    assert rel_l2(d, ref) <= 1e-5
    # in place: the caller's gradient becomes the direction
    opt.direction(gd, gd)
    assert np.array_equal(gd.cpu().numpy(), d)
    opt.close()
