"""Energy and gradient from one pass over the attraction's pairs, in every tile
shape and fold, against the oracle, and the autograd function on top of it.

Gates: those of the separate calls -- (A - R) within 1e-5 relative L2 (times
the condition number of the subtraction) and 1e-5 absolute, F^a and F^r within
1e-6 -- and the two passes against the one: same FP32 terms, sums grouped
differently, 2e-6.
"""
import numpy as np
import pytest

import inputs
import oracle
from gpu_util import GRAD_ABS, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2108_02991_gb300 as sp
    return sp


def problem(N, seed, dt=np.float32):
    rng = np.random.default_rng(seed)
    K = (0.35 * rng.normal(size=(N, 3))).clip(-0.5, 0.5).astype(np.float32)
    n = [(13, 9, 7), (64, 20, 6), (1, 5, 3)][seed % 3]
    rho = rng.uniform(0.0, 1.0, size=(n[2], n[1], n[0]))
    return K.astype(dt), inputs.Grid(n, -0.5, 0.5, (rho / rho.sum()).astype(np.float32))


@pytest.mark.parametrize("acc", [0, 1])
@pytest.mark.parametrize("shape", [0, 1, 2])
@pytest.mark.parametrize("N,eps,dt", [(2, 0.0, np.float32), (1025, 0.02, np.float64),
                                      (3000, 0.0, np.float32)])
def test_every_shape_against_the_oracle(sp, N, eps, dt, shape, acc):
    K, grid = problem(N, N + shape, dt)
    c = sp.sparkling_create(0)
    try:
        sp.sparkling_set_shape(c, "attraction", shape)
        sp.sparkling_set_regularisation(c, eps)
        g = sp.make_grid(torch.from_numpy(grid.rho).cuda(), grid.lo, grid.hi, grid.n)
        (F, Fa, Fr), dK = sp.sparkling_energy_and_grad(c, torch.from_numpy(K).cuda(), g, acc)
    finally:
        c.close()
    A0, R0, G0 = oracle.forces(K.astype(np.float64), grid, eps=eps)
    _, Fa0, Fr0 = oracle.energy(K.astype(np.float64), grid, eps=eps)
    assert Fa == pytest.approx(Fa0, rel=1e-6) and Fr == pytest.approx(Fr0, rel=1e-6)
    assert F == Fa - Fr
    G = dK.cpu().numpy() * N
    cond = (np.linalg.norm(A0) + np.linalg.norm(R0)) / np.linalg.norm(G0) / 2
    assert rel_l2(G, G0) < 1e-5 * max(cond, 1.0)
    np.testing.assert_allclose(G, G0, rtol=0, atol=GRAD_ABS)


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_autograd_is_the_separate_calls(sp, dt):
    """25000 samples (the symmetric repulsion): value and gradient equal the
    separate calls'; scaled loss, repeated backward, no gradient asked for."""
    Kn, grid = problem(25000, 5)
    c = sp.sparkling_create(0)
    try:
        rho = torch.from_numpy(grid.rho).cuda()
        g = sp.make_grid(rho, grid.lo, grid.hi, grid.n)
        K = torch.from_numpy(Kn).cuda().to(dt).requires_grad_(True)
        F = sp.sparkling_energy_fn(K, rho, c)
        (a,) = torch.autograd.grad(3.0 * F, K, retain_graph=True)
        (b,) = torch.autograd.grad(F, K)
        F0 = sp.sparkling_energy(c, K.detach(), g)[0]
        d = sp.sparkling_energy_backward(c, K.detach(), g)
        assert a.dtype == dt and float(F.detach()) == pytest.approx(F0, rel=2e-6)
        assert rel_l2(b.cpu().numpy(), d.cpu().numpy()) < 2e-6
        assert rel_l2(a.cpu().numpy(), 3.0 * b.cpu().numpy()) < 2e-7
        assert not b.requires_grad
        with torch.no_grad():
            assert not sp.sparkling_energy_fn(K, rho, c).requires_grad
        assert not sp.sparkling_energy_fn(K.detach(), rho, c).requires_grad
        # in-place change between forward and backward is still noticed
        L = K * 1.0
        F = sp.sparkling_energy_fn(L, rho, c)
        L += 1.0
        with pytest.raises(RuntimeError):
            F.backward()
    finally:
        c.close()


def test_fast_modes_leave_the_gradient_to_the_backward(sp):
    Kn, grid = problem(3000, 6)
    c = sp.sparkling_create(0)
    try:
        sp.sparkling_set_repulsion(c, sp.REPULSION_MESH, sp.make_mesh(24))
        rho = torch.from_numpy(grid.rho).cuda()
        g = sp.make_grid(rho, grid.lo, grid.hi, grid.n)
        K = torch.from_numpy(Kn).cuda().requires_grad_(True)
        E, dK = sp.sparkling_energy_and_grad(c, K.detach(), g)
        assert dK is None and E == sp.sparkling_energy(c, K.detach(), g)
        (b,) = torch.autograd.grad(sp.sparkling_energy_fn(K, rho, c), K)
        assert torch.equal(b, sp.sparkling_energy_backward(c, K.detach(), g))
    finally:
        c.close()
