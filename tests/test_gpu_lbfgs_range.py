"""l-BFGS inner products of vectors that are large where the other is small, so that every product is far
below the product of the two largest elements; directions written over the gradient they are made from."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbfgs():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2305_14130_gb300.optim import LBFGS
    return LBFGS


def dev(n, head):
    a = np.zeros(n, np.float32)
    a[:len(head)] = head
    return torch.tensor(a, device="cuda")


# s^T y comes from a tiny element of s alone.  Where s and y are zero, d = -gamma g with
# gamma = s^T y / y^T y, rounded to FP32 once.
@pytest.mark.parametrize("s,y", [((1e20, 3e-26), (0.0, 1.0)), ((1e25, 1e-25), (0.0, 1e12)), ((1e-6, 2e-40), (0.0, 1e-10))])
@pytest.mark.parametrize("n", [8, 3001])
def test_curvature_of_a_pair_of_opposite_magnitudes(lbfgs, n, s, y):
    s64, y64 = np.float32(s).astype(np.float64), np.float32(y).astype(np.float64)
    opt = lbfgs(n, m=1)
    assert opt.push(dev(n, s), dev(n, y))
    d = opt.direction(dev(n, (0.0, 0.0, 1.0)))
    assert abs(d[2].item() / -(s64 @ y64 / (y64 @ y64)) - 1) <= 2.0 ** -23
    opt.close()


@pytest.mark.parametrize("n", [8, 3001])
def test_coefficient_of_a_gradient_of_opposite_magnitude(lbfgs, n):
    # s^T y = 2, y^T y = 1, gamma = 2; s^T g = 1 from the tiny element of s: alpha = 1/2, beta = -1/2
    opt = lbfgs(n, m=1)
    assert opt.push(dev(n, (1e19, 1e-27, 1.0)), dev(n, (1e-19, 0.0, 1.0)))
    d = opt.direction(dev(n, (0.0, 1e27, 0.0))).cpu().numpy()
    # a few FP32 roundings of s, y, g and of each update
    assert np.allclose(d[:2], (-1e19, -2e27), rtol=2.0 ** -20, atol=0) and abs(d[2]) <= 2.0 ** -20
    opt.close()


@pytest.mark.parametrize("pairs", [0, 1])
@pytest.mark.parametrize("shift", [-5, 4, 70_000])
def test_direction_over_part_of_its_gradient(lbfgs, pairs, shift):
    n = 3_000_000
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    buf = torch.randn(n + abs(shift), generator=gen, device="cuda")
    g = buf[max(-shift, 0):][:n]
    d = buf[max(shift, 0):][:n]
    opt = lbfgs(n, m=1)
    for _ in range(pairs):
        s = torch.randn(n, generator=gen, device="cuda")
        assert opt.push(s, 2 * s)
    ref = opt.direction(g.clone())
    opt.direction(g, d)
    assert torch.equal(d, ref)
    opt.close()
