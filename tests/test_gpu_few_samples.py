"""Gradient and energy of few samples: the directed repulsion over the whole
GPU (64 targets a warp, slices of the sources), its boundary to the symmetric
kernel, and the slot sums of eight threads a sample.

Gates: A and R within the accumulation bound of every gradient test (1e-5
relative L2 and absolute), the energy terms within 1e-6; on both sides of the
boundary both kernels give the same sums up to FP32 rounding (2e-6 relative
L2: sums of at most 1024 unit vectors, ~sqrt(1024) 2^-24).
"""
import numpy as np
import pytest

import inputs
import oracle
from gpu_util import assert_grad_close, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2108_02991_gb300 as sp
    return sp


def evaluate(sp, ctx, K, grid, dt, acc=0):
    Kd = torch.from_numpy(K.astype(dt)).cuda()
    g = sp.make_grid(torch.from_numpy(grid.rho).cuda(), grid.lo, grid.hi, grid.n)
    A = torch.empty(K.shape, dtype=torch.float64, device="cuda")
    R, G = torch.empty_like(A), torch.empty_like(A)
    sp.sparkling_grad(ctx, Kd, g, acc, G=G, A=A, R=R)
    sp.sparkling_status(ctx)
    F = sp.sparkling_energy(ctx, Kd, g, acc)
    return A.cpu().numpy(), R.cpu().numpy(), G.cpu().numpy(), F


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("eps", [0.0, 0.02])
@pytest.mark.parametrize("N", [2, 3, 31, 33, 63, 64, 65, 129, 1000, 1024, 1025, 2500, 4100])
def test_against_the_oracle(sp, N, eps, dt):
    rng = np.random.default_rng(N)
    K = rng.uniform(-0.5, 0.5, size=(N, 3)).astype(np.float32)
    if N > 3:
        K[1] = K[0]
    n = [(9, 7, 5), (16, 16, 16), (1, 3, 2)][N % 3]
    rho = rng.uniform(0.5, 1.5, size=(n[2], n[1], n[0]))
    grid = inputs.Grid(n, -0.5, 0.5, (rho / rho.sum()).astype(np.float32))
    c = sp.sparkling_create(0)
    try:
        sp.sparkling_set_regularisation(c, eps)
        A, R, G, (F, Fa, Fr) = evaluate(sp, c, K, grid, dt, acc=N % 2)
    finally:
        c.close()
    K64 = K.astype(np.float64)
    A0, R0, _ = oracle.forces(K64, grid, eps=eps)
    _, Fa0, Fr0 = oracle.energy(K64, grid, eps=eps)
    assert_grad_close(A, A0, "A")
    assert_grad_close(R, R0, "R")
    np.testing.assert_allclose(G, A - R, rtol=0, atol=1e-15)
    assert Fa == pytest.approx(Fa0, rel=1e-6)
    assert Fr == pytest.approx(Fr0, rel=1e-6)


@pytest.mark.parametrize("N", [20480, 20481])
def test_boundary_to_the_symmetric_kernel(sp, N):
    K = np.random.default_rng(N).uniform(-0.5, 0.5, size=(N, 3)).astype(np.float32)
    grid = inputs.density_gaussian(8, 0.2)
    a, b = sp.sparkling_create(0), sp.sparkling_create(0)
    try:
        sp.sparkling_set_shape(b, "repulsion", 3)          # the symmetric kernel at every size
        A, R, _, F = evaluate(sp, a, K, grid, np.float32)
        A1, R1, _, F1 = evaluate(sp, b, K, grid, np.float32)
        again = evaluate(sp, a, K, grid, np.float32)
    finally:
        a.close()
        b.close()
    assert rel_l2(R, R1) < 2e-6
    assert F[2] == pytest.approx(F1[2], rel=1e-6)
    np.testing.assert_array_equal(again[1], R)             # order-free sums
    np.testing.assert_array_equal(again[0], A)
    assert again[3] == F
