"""Short-range pairs of the fast repulsion through clusters of sorted samples:
counts around the cluster (32), the group (64) and the boxes' levels (1024,
32768), samples that crowd, coincide or lie on lines through the centre.

Gate: the library's FP32 arithmetic against the same split summed in FP64 --
the oracle's exact short-range sum plus the NumPy restatement of the mesh's
long-range part -- so that the mesh's method error (up to 5e-5 of R where
samples crowd at 24 cells) drops out: 1e-6 relative L2 and 2e-6 absolute on R
(2e-6 relative on F^r), from the 1.5e-7 of the erfc, ~1e-7 of sums of at most
4096 FP32 terms and a few 1e-7 of the FP32 transforms.
"""
import numpy as np
import pytest

import inputs
import mesh_reference as p3m
import oracle
from gpu_util import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SPEC = p3m.MeshSpec(n_cells=24, sigma=2.5 / 24, guard=4)       # 32 mesh cells an axis


@pytest.fixture(scope="module")
def sp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2108_02991_gb300 as sp
    return sp


@pytest.fixture(scope="module")
def ctxs(sp):
    direct, mesh = sp.sparkling_create(0), sp.sparkling_create(0)
    sp.sparkling_set_repulsion(mesh, sp.REPULSION_MESH, sp.make_mesh(24))
    yield direct, mesh
    direct.close()
    mesh.close()


def samples(kind, N):
    rng = np.random.default_rng(N)
    if kind == "uniform":
        return rng.uniform(-0.5, 0.5, size=(N, 3))
    if kind == "crowded":            # half of them inside one cell of the mesh
        K = rng.uniform(-0.5, 0.5, size=(N, 3))
        K[::2] = 0.1 + 0.01 * rng.uniform(-1, 1, size=K[::2].shape)
        return K
    u = inputs.hemisphere_directions(max(N // 64, 1))
    return (u[np.arange(N) % u.shape[0]] * rng.uniform(-0.5, 0.5, size=(N, 1)))


def evaluate(sp, ctx, K, g):
    G, R = torch.empty(K.shape, dtype=torch.float64, device="cuda"), torch.empty(
        K.shape, dtype=torch.float64, device="cuda")
    sp.sparkling_grad(ctx, K, g, G=G, R=R)
    sp.sparkling_status(ctx)
    return R.cpu().numpy(), sp.sparkling_energy(ctx, K, g)[2]


@pytest.mark.parametrize("kind", ["uniform", "crowded", "spokes"])
@pytest.mark.parametrize("N", [31, 32, 33, 63, 64, 65, 127, 129, 1023, 1025, 2049, 32769, 70000])
def test_against_the_split_in_fp64(sp, ctxs, N, kind):
    K = samples(kind, N).astype(np.float32)
    if N > 40:
        K[5] = K[40]                               # a coincident pair
    grid = inputs.density_gaussian(4, 0.2)
    g = sp.make_grid(torch.from_numpy(grid.rho).cuda(), grid.lo, grid.hi, grid.n)
    Kd = torch.from_numpy(K).cuda()
    R, Fr = evaluate(sp, ctxs[1], Kd, g)
    K64 = K.astype(np.float64)
    S, _, eS, _ = oracle.repulsion_split(K64, SPEC.sigma, rc=4.0 * SPEC.sigma)
    Lm, eLm = p3m.mesh_long(K64, SPEC)
    want = (S + Lm) / N
    assert rel_l2(R, want) < 1e-6
    np.testing.assert_allclose(R, want, rtol=0, atol=2e-6)
    # pairs at distance 0 (every sample with itself, and the coincident pair,
    # which the oracle's sum leaves out) count g_short(0) = -sigma / sqrt(pi)
    zeros = N + (2 if N > 40 else 0)
    er = eS.sum() - zeros * SPEC.sigma / np.sqrt(np.pi) + eLm.sum()
    assert Fr == pytest.approx(er / (2.0 * N * N), rel=2e-6)


@pytest.mark.parametrize("hi,rc_sigmas", [(0.5, 2.5), (0.5, 6.0), (500.0, 4.0), (5e-4, 4.0)])
def test_cut_offs_and_units(sp, hi, rc_sigmas):
    """A short and a long cut-off, and boxes of other units (the coordinates
    are scaled by a power of two inside): R scales with nothing."""
    K = (samples("uniform", 1500) * 2 * hi).astype(np.float32)
    rho = torch.full((2, 2, 2), 0.125, device="cuda")
    g = sp.make_grid(rho, -hi, hi)
    Kd = torch.from_numpy(K).cuda()
    direct, mesh = sp.sparkling_create(0), sp.sparkling_create(0)
    try:
        sp.sparkling_set_repulsion(mesh, sp.REPULSION_MESH, sp.make_mesh(24, 2.5, rc_sigmas, -hi, hi))
        R0, Fr0 = evaluate(sp, direct, Kd, g)
        R, Fr = evaluate(sp, mesh, Kd, g)
    finally:
        direct.close()
        mesh.close()
    # erfc(2.5) = 4.1e-4 of the pairs just beyond a short cut-off is missing
    bound = 1e-5 if rc_sigmas >= 4 else 1e-3
    assert rel_l2(R, R0) < bound
    assert Fr == pytest.approx(Fr0, rel=2 * bound)
