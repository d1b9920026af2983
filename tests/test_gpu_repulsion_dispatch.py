"""Where the repulsion goes over from the directed to the symmetric kernel, and
the symmetric kernel with fewer tile pairs than the GPU holds CTAs.

Gates: both kernels' sums agree to FP32 rounding (2e-6 relative L2, energy
1e-6, as in test_gpu_few_samples.py).  The gates of the times leave a factor of
1.2 and more to the measured ratios.
"""
import numpy as np
import pytest

import inputs
from gpu_util import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2108_02991_gb300 as sp
    return sp


def problem(sp, N):
    K = torch.rand(N, 3, device="cuda", generator=torch.Generator("cuda").manual_seed(N)) - 0.5
    rho = torch.from_numpy(inputs.density_gaussian(8, 0.2).rho).cuda()
    return K, sp.make_grid(rho)


def context(sp, shape=None):
    c = sp.sparkling_create(0)
    if shape is not None:
        sp.sparkling_set_shape(c, "repulsion", shape)
    return c


def repulsion(sp, c, K, g, eps=0.0):
    R = torch.empty_like(K, dtype=torch.float64)
    sp.sparkling_set_regularisation(c, eps)
    sp.sparkling_grad(c, K, g, 0, R=R)
    sp.sparkling_status(c)
    return R.cpu().numpy(), sp.sparkling_energy(c, K, g)[2]


@pytest.mark.parametrize("eps", [0.0, 0.02])
@pytest.mark.parametrize("N", [11263, 11264, 11265, 12288, 16384, 16385, 17409, 24577])
def test_both_sides_of_the_rules(sp, N, eps):
    """11264: directed below; 16385: more tile pairs (153) than SMs."""
    K, g = problem(sp, N)
    a, b = context(sp), context(sp, 0)
    try:
        R, F = repulsion(sp, a, K, g, eps)
        R1, F1 = repulsion(sp, b, K, g, eps)
        assert rel_l2(R, R1) < 2e-6
        assert F == pytest.approx(F1, rel=1e-6)
        np.testing.assert_array_equal(repulsion(sp, a, K, g, eps)[0], R)
    finally:
        a.close()
        b.close()


@pytest.mark.parametrize("shape", [0, 1, 2, 3])
@pytest.mark.parametrize("N", [2, 1024, 1025, 5000])
def test_fewer_tile_pairs_than_ctas(sp, N, shape):
    K, g = problem(sp, N)
    a, b = context(sp), context(sp, shape)
    try:
        R, F = repulsion(sp, a, K, g)
        R1, F1 = repulsion(sp, b, K, g)
        assert rel_l2(R1, R) < 2e-6
        assert F1 == pytest.approx(F, rel=1e-6)
    finally:
        a.close()
        b.close()


def repulsion_us(sp, c, call, reps=8):
    call()
    call()
    sp.sparkling_set_timing(c, True)
    sp.sparkling_kernel_times(c, reset=True)
    for _ in range(reps):
        call()
    torch.cuda.synchronize()
    t = sp.sparkling_kernel_times(c, reset=True)["repulsion"]
    sp.sparkling_set_timing(c, False)
    return 1e3 * t[0] / t[1]


@pytest.mark.parametrize("N", [4096, 10240, 13312, 20480])
def test_the_rule_takes_the_faster_kernel(sp, N):
    """At most 1.15 times the best symmetric shape, for the force and the
    energy (directed up to 20480 samples: 1.2 and 1.5 times at the last two)."""
    K, g = problem(sp, N)
    G = torch.empty_like(K)
    times = []
    for shape in (None, 0, 1, 2, 3):
        c = context(sp, shape)
        try:
            times.append((repulsion_us(sp, c, lambda: sp.sparkling_grad(c, K, g, 0, G)),
                          repulsion_us(sp, c, lambda: sp.sparkling_energy(c, K, g))))
        finally:
            c.close()
    for mine, best in zip(times[0], np.min(times[1:], axis=0)):
        assert mine < 1.15 * best + 2.0


def test_a_tile_pair_has_an_sm_to_itself(sp):
    """36 and 55 tile pairs take the time of one, not of two on an SM (the
    former took 1.9 times the latter)."""
    t = []
    for N in (8192, 10240):
        K, g = problem(sp, N)
        G = torch.empty_like(K)
        c = context(sp, 3)
        try:
            t.append(repulsion_us(sp, c, lambda: sp.sparkling_grad(c, K, g, 0, G)))
        finally:
            c.close()
    assert t[0] < 1.3 * t[1]
