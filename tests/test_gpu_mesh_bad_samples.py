"""The fast repulsion with a sample that is not a number, infinite or far outside
the mesh: the call reports it, and the other samples' sums are those without it.

Gate: 1e-6 relative L2, the FP32 sums in another grouping (a few 1e-7).
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


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf"), 1e30, 3.0])
@pytest.mark.parametrize("N", [40, 1000, 5000])
def test_the_other_samples_are_not_spoilt(sp, N, bad):
    K = np.random.default_rng(N).uniform(-0.5, 0.5, size=(N, 3)).astype(np.float32)
    g = inputs.density_gaussian(4, 0.2)
    rho = torch.from_numpy(g.rho).cuda()
    grid = sp.make_grid(rho, g.lo, g.hi, g.n)
    c = sp.sparkling_create(0)
    try:
        sp.sparkling_set_repulsion(c, sp.REPULSION_MESH, sp.make_mesh(24))
        at = N // 2
        rest = np.delete(np.arange(N), at)
        R = torch.empty(N, 3, dtype=torch.float64, device="cuda")
        Kb = K.copy()
        Kb[at, 1] = bad
        sp.sparkling_grad(c, torch.from_numpy(Kb).cuda(), grid, R=R, G=torch.empty_like(R))
        with pytest.raises(sp.SparklingError) as e:
            sp.sparkling_status(c)
        assert e.value.code == (sp.E_RANGE if np.isfinite(bad) else sp.E_NONFINITE)
        W = torch.empty(N - 1, 3, dtype=torch.float64, device="cuda")
        sp.sparkling_grad(c, torch.from_numpy(K[rest]).cuda(), grid, R=W, G=torch.empty_like(W))
        sp.sparkling_status(c)
    finally:
        c.close()
    assert rel_l2(R.cpu().numpy()[rest] * N, W.cpu().numpy() * (N - 1)) < 1e-6
