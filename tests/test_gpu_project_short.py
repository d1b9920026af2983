"""Many short shots: the violations asked for beside a projection, and the FP64
projection's shapes.

Gates of the results as in test_gpu_project_reg.py (FP64 1e-11, FP32 one ulp of
1/2).  Gates of the times compare two calls on the same GPU and leave a factor
of 1.3 and more to what is expected.
"""
import numpy as np
import pytest

import oracle
from gpu_util import PROJ_F32_ROUND

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2108_02991_gb300 as sp
    return sp


@pytest.fixture(scope="module")
def ctx(sp):
    c = sp.sparkling_create(0)
    yield c
    c.close()


def shots(Nc, Ns, dt):
    rng = np.random.default_rng(Nc + Ns)
    K = np.cumsum(rng.normal(scale=0.02, size=(Nc, Ns, 3)), axis=1)
    return np.clip(K + rng.uniform(-0.4, 0.4, size=(Nc, 1, 3)), -0.6, 0.6).reshape(-1, 3).astype(dt)


def radii(Ns):
    return 1.0 / (2 * Ns), 1.0 / (8 * Ns * Ns)


def project_ms(sp, ctx, Nc, Ns, dt, n_iter, viol=False, reps=5):
    K0 = torch.from_numpy(shots(Nc, Ns, dt)).cuda()
    K = K0.clone()
    pr = sp.make_proj(*radii(Ns), 0.5, n_iter)
    sp.sparkling_project(ctx, K, Nc, Ns, pr, want_violation=viol)
    sp.sparkling_set_timing(ctx, True)
    sp.sparkling_kernel_times(ctx, reset=True)
    for _ in range(reps):
        K.copy_(K0)
        sp.sparkling_project(ctx, K, Nc, Ns, pr, want_violation=viol)
    torch.cuda.synchronize()
    t = sp.sparkling_kernel_times(ctx, reset=True)["project"]
    sp.sparkling_set_timing(ctx, False)
    return t[0] / t[1]


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("Nc,Ns", [(1, 1), (700, 1), (300, 2), (1, 3), (4000, 3), (40, 255), (41, 256), (40, 257),
                                   (3, 9000)])
def test_violations_of_every_sample(sp, ctx, Nc, Ns, dt):
    """The four maxima of the result as written, pin on the last sample: blocks
    that hold many shots, end inside one, and shots longer than a block."""
    K = torch.from_numpy(shots(Nc, Ns, dt)).cuda()
    a, b = radii(Ns)
    pr = sp.make_proj(a, b, 0.5, 3, Ns - 1, (0.1, -0.2, 0.3))
    v = sp.sparkling_project(ctx, K, Nc, Ns, pr, want_violation=True)
    s = K.cpu().numpy().astype(np.float64).reshape(Nc, Ns, 3)
    d1 = np.linalg.norm(np.diff(s, axis=1), axis=2)
    d2 = np.linalg.norm(s[:, 2:] - 2.0 * s[:, 1:-1] + s[:, :-2], axis=2)
    want = [max(d1.max(initial=0.0) - a, 0.0), max(d2.max(initial=0.0) - b, 0.0),
            max(np.abs(s).max() - 0.5, 0.0), np.abs(s[:, -1] - [0.1, -0.2, 0.3]).max()]
    np.testing.assert_allclose(v, want, rtol=1e-12, atol=1e-15)


@pytest.mark.parametrize("dt", [np.float32, np.float64])
def test_violations_cost_little(sp, ctx, dt):
    """A pass over the result beside an iteration that reads and writes it: at
    most three times the projection alone (a block a shot took ten times)."""
    assert (project_ms(sp, ctx, 20000, 2, dt, 1, viol=True) <
            3.0 * project_ms(sp, ctx, 20000, 2, dt, 1) + 0.02)


def check(sp, ctx, Nc, Ns, dt, n_iter, pin_index=-1):
    K = shots(Nc, Ns, dt)
    a, b = radii(Ns)
    ref = oracle.project(K.astype(np.float64), Nc, Ns, a, b, box=0.5, pin_index=pin_index, n_iter=n_iter)
    ref = ref[0] if isinstance(ref, tuple) else ref
    Kd = torch.from_numpy(K).cuda()
    sp.sparkling_project(ctx, Kd, Nc, Ns, sp.make_proj(a, b, 0.5, n_iter, pin_index))
    if dt == np.float64:
        np.testing.assert_allclose(Kd.cpu().numpy(), ref, rtol=0, atol=1e-11)
    else:
        np.testing.assert_allclose(Kd.cpu().numpy(), ref.astype(np.float32), rtol=0, atol=PROJ_F32_ROUND)


@pytest.mark.parametrize("Nc,Ns", [(400, 1), (400, 2), (153, 31), (700, 32), (700, 33), (300, 65), (300, 96),
                                   (160, 160), (153, 255), (153, 257), (160, 767), (153, 769)])
def test_more_fp64_shots_than_sms(sp, ctx, Nc, Ns):
    check(sp, ctx, Nc, Ns, np.float64, 25, pin_index=Ns - 1)


@pytest.mark.parametrize("n_iter", [0, 1, 100])
@pytest.mark.parametrize("dt", [np.float32, np.float64])
def test_lone_samples_are_clipped(sp, ctx, dt, n_iter):
    K = torch.from_numpy(shots(500, 1, dt)).cuda()
    want = K.clamp(-0.5, 0.5)
    sp.sparkling_project(ctx, K, 500, 1, sp.make_proj(*radii(1), 0.5, n_iter))
    assert torch.equal(K, want)


def test_fp64_times_follow_the_samples(sp, ctx):
    """Bound by the FP64 pipe, which half a warp occupies like a whole one:
    shots of 32 samples take one warp of one sample a thread (72 units an
    iteration) where 33 samples take one of two (122), expected 0.6, gate 0.8
    (it was 1.0); lone samples have no iteration to do."""
    t = {n: project_ms(sp, ctx, 20000, n, np.float64, 100) for n in (1, 2, 32, 33)}
    assert t[32] < 0.8 * t[33]
    assert t[1] < 0.2 * t[2]
