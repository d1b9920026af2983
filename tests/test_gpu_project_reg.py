"""The projection with its state in registers, at the edges of its shapes.

FP32 samples iterate in two-float arithmetic (hi + lo, 48 bits), FP64 samples
in FP64; a thread owns one or two samples, a warp 32 or 64, a CTA up to 512
(FP32) or 1024 (FP64), longer shots a cluster of up to eight CTAs.  Gates: the
FP64 iterates agree with the oracle's to 1e-11; an FP32 result is the oracle's
rounded one up to one ulp of 1/2 (2^-24), since the two-float iteration's own
error (~2^-45 of the duals) can only flip the last rounding.
"""
import numpy as np
import pytest

import inputs
import oracle
from gpu_util import GRAD_ABS, PROJ_F32_ROUND

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


def shots(Nc, Ns, seed, spread):
    rng = np.random.default_rng(seed)
    K = np.cumsum(rng.normal(scale=spread, size=(Nc, Ns, 3)), axis=1)
    return np.clip(K + rng.uniform(-0.45, 0.45, size=(Nc, 1, 3)), -0.6, 0.6).reshape(-1, 3)


def check(sp, ctx, K, Nc, Ns, dt, alpha, beta, n_iter, box=0.5, pin_index=-1, pin=(0, 0, 0)):
    K = K.astype(dt)
    ref = oracle.project(K.astype(np.float64), Nc, Ns, alpha, beta, box=box, pin_index=pin_index,
                         pin=pin, n_iter=n_iter)
    ref = ref[0] if isinstance(ref, tuple) else ref
    Kd = torch.from_numpy(K.copy()).cuda()
    sp.sparkling_project(ctx, Kd, Nc, Ns, sp.make_proj(alpha, beta, box, n_iter, pin_index, pin))
    sp.sparkling_status(ctx)
    out = Kd.cpu().numpy()
    if dt == np.float64:
        np.testing.assert_allclose(out, ref, rtol=0, atol=1e-11)
    else:
        np.testing.assert_allclose(out, ref.astype(np.float32), rtol=0, atol=PROJ_F32_ROUND)


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("Ns", [1, 2, 3, 31, 32, 33, 64, 65, 127, 128, 129, 256, 257, 511, 512, 513,
                                1024, 1025, 1537, 4095, 4097, 8192, 8193])
def test_warp_cta_and_cluster_edges(sp, ctx, Ns, dt):
    """Every edge of the split of a shot over warps, CTAs and clusters (8193:
    past it, the form with its state in memory); box active, pin on an edge."""
    a, b = 1.0 / (2 * Ns), 1.0 / (8 * Ns * Ns)
    K = shots(3, Ns, Ns, 4.0 * a)
    pin_index = min(Ns - 1, 64) if Ns % 2 else -1
    check(sp, ctx, K, 3, Ns, dt, a, b, 40, pin_index=pin_index, pin=(0.0, 0.125, -0.25))


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("kw", [dict(alpha=float("inf"), beta=1e-5), dict(alpha=2e-3, beta=float("inf")),
                                dict(alpha=1e-14, beta=1e-16), dict(alpha=3.0, beta=5.0),
                                dict(alpha=2e-3, beta=1e-5, n_iter=0),
                                dict(alpha=2e-3, beta=1e-5, n_iter=1),
                                dict(alpha=2e-3, beta=1e-5, box=0.1)])
def test_radii_boxes_and_iteration_counts(sp, ctx, kw, dt):
    """Constraints switched off, radii below the two-float form's range, an
    inactive set (the result is the clipped input), no iteration and one."""
    kw = dict(dict(n_iter=60), **kw)
    K = shots(5, 150, 7, 5e-3)
    check(sp, ctx, K, 5, 150, dt, kw.pop("alpha"), kw.pop("beta"), kw.pop("n_iter"), **kw)


def test_more_iterations_than_the_momentum_table(sp, ctx):
    check(sp, ctx, shots(5, 150, 7, 5e-3), 5, 150, np.float32, 2e-3, 1e-5, 4200)


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("Nc,Ns,n_iter", [(1, 96, 1), (1, 97, 2), (1, 300, 37), (2, 512, 100), (5, 777, 64),
                                          (7, 1000, 100), (18, 500, 60), (37, 129, 100), (76, 130, 33),
                                          (3, 2560, 60), (1, 4095, 50), (2, 8190, 30)])
def test_few_shots_over_many_ctas(sp, ctx, Nc, Ns, n_iter, dt):
    """Shots split over CTAs that also compute a halo of their neighbours:
    owners' bands, copies every few iterations, none at all, pins in a halo."""
    a, b = 1.0 / (2 * Ns), 1.0 / (8 * Ns * Ns)
    check(sp, ctx, shots(Nc, Ns, Nc + Ns, 4.0 * a), Nc, Ns, dt, a, b, n_iter, pin_index=Ns // 2)


def test_more_shots_than_a_grid_holds_at_once(sp, ctx):
    check(sp, ctx, shots(1500, 33, 3, 0.02), 1500, 33, np.float32, 1 / 66, 1 / 8712, 30)


@pytest.mark.parametrize("Ns", [1, 96, 700])
def test_batched_projections_after_the_engine(sp, ctx, Ns):
    """FP32 trajectories of uneven size whose shots take one warp, one CTA and
    a cluster, against the oracle step; own radii, pins and iteration counts."""
    rng = np.random.default_rng(Ns)
    counts = [2, 5, 3]
    g = inputs.density_gaussian(8, 0.2, 0.1)
    rho = torch.from_numpy(g.rho).cuda()
    Ks, grids, projs, etas, refs = [], [], [], [], []
    for b, c in enumerate(counts):
        a, be = (0.5 + b) / (2 * Ns), (0.5 + b) / (8 * Ns * Ns)
        K = shots(c, Ns, 10 * Ns + b, 2.0 * a).astype(np.float32)
        eta, n_iter, pin = 0.05 / (c * Ns), 20 + 10 * b, Ns // 2 if b else -1
        Ks.append(K)
        grids.append(sp.make_grid(rho, g.lo, g.hi, g.n))
        projs.append(sp.make_proj(a, be, 0.5, n_iter, pin))
        etas.append(eta)
        refs.append(oracle.step(K.astype(np.float64), c, Ns, g, eta, a, be, 0.5, pin,
                                (0.0, 0.0, 0.0), n_iter))
    off = np.concatenate([[0], np.cumsum([k.shape[0] for k in Ks])])
    for one in (True, False):
        K = torch.from_numpy(np.concatenate(Ks)).cuda()
        sp.sparkling_step_batched(ctx, K, off, Ns, grids, etas, projs, one_launch=one, graph=False)
        sp.sparkling_status(ctx)
        out = K.cpu().numpy()
        for b in range(len(Ks)):
            np.testing.assert_allclose(out[off[b]:off[b + 1]], refs[b].astype(np.float32), rtol=0,
                                       atol=PROJ_F32_ROUND + 4 * etas[b] * GRAD_ABS)
