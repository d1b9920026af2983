"""Which arithmetic a projection of FP32 samples runs in: two-float sums by
default, FP64 where the context asks for it, and outside the two-float form's
range FP64 or (opt-in) the FP32 iteration on the displacement -- in
sparkling_project and as projection items of the batched engine.

Gates: FP64 and two-float results are the oracle's rounded ones up to one ulp of
1/2 (PROJ_F32_ROUND); the mixed form has its own bound (proj_tol_f32); a step
adds 4 eta times the gradient's error, as in test_gpu_batched.py.
"""
import numpy as np
import pytest

import inputs
import oracle
from gpu_util import GRAD_ABS, PROJ_F32_ROUND, proj_tol_f32

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2108_02991_gb300 as sp
    return sp


@pytest.fixture
def ctx(sp):
    c = sp.sparkling_create(0)
    yield c
    c.close()


def shots(Nc, Ns, seed, spread=0.02):
    rng = np.random.default_rng(seed)
    K = np.cumsum(rng.normal(scale=spread, size=(Nc, Ns, 3)), axis=1)
    return np.clip(K + rng.uniform(-0.4, 0.4, size=(Nc, 1, 3)), -0.5, 0.5).reshape(-1, 3).astype(np.float32)


@pytest.mark.parametrize("c", [0.11, 0.25, 0.3, 0.37])
def test_fp64_asked_for_is_fp64(sp, ctx, c):
    """One row of length c and a radius of c (1 - 2^-42): the first sample moves
    by ~c 2^-43.  FP64 has it to 2^-53 of the dual, ten times in the fixed point's
    sum: within c 2^-49.  It also needs the state that the two-float form keeps in
    registers."""
    c = float(np.float32(c))
    a = c * (1.0 - 2.0 ** -42)
    K = np.zeros((2, 3), np.float32)
    K[1, 2] = c
    ref = oracle.project(K.astype(np.float64), 1, 2, a, float("inf"), n_iter=300)
    sp.sparkling_set_projection(ctx, sp.PROJECTION_FP64)
    Kd = torch.from_numpy(K).cuda()
    sp.sparkling_project(ctx, Kd, 1, 2, sp.make_proj(a, float("inf"), 0.5, 300))
    out = Kd.cpu().numpy().astype(np.float64)
    assert ref[0, 2] > c * 2.0 ** -45
    np.testing.assert_allclose(out[0], ref[0], rtol=0, atol=c * 2.0 ** -49)

    sp.sparkling_set_memory_limit(ctx, 1)
    Kd = torch.from_numpy(shots(1, 2560, 1)).cuda()
    pr = sp.make_proj(1e-3, 1e-5, 0.5, 2)
    with pytest.raises(sp.SparklingError) as e:
        sp.sparkling_project(ctx, Kd, 1, 2560, pr)
    assert e.value.code == sp.E_NOMEM
    sp.sparkling_set_projection(ctx, sp.PROJECTION_DEFAULT)
    sp.sparkling_project(ctx, Kd, 1, 2560, pr)


@pytest.mark.parametrize("Nc,Ns,n_iter,pin", [(5, 1, 7, 0), (9, 33, 40, 32), (200, 64, 30, -1), (3, 700, 60, 350)])
def test_fp64_asked_for_against_the_oracle(sp, ctx, Nc, Ns, n_iter, pin):
    K = shots(Nc, Ns, Ns)
    a, b = 1.0 / (2 * Ns), 1.0 / (8 * Ns * Ns)
    ref = oracle.project(K.astype(np.float64), Nc, Ns, a, b, pin_index=pin, pin=(0.1, 0.0, -0.1), n_iter=n_iter)
    sp.sparkling_set_projection(ctx, sp.PROJECTION_FP64)
    Kd = torch.from_numpy(K).cuda()
    sp.sparkling_project(ctx, Kd, Nc, Ns, sp.make_proj(a, b, 0.5, n_iter, pin, (0.1, 0.0, -0.1)))
    np.testing.assert_allclose(Kd.cpu().numpy(), ref.astype(np.float32), rtol=0, atol=PROJ_F32_ROUND)
