"""The register form of the projection at the ends of its numbers: rows that
barely leave their ball, and samples that are huge, tiny or not numbers."""
import numpy as np
import pytest

import inputs
import oracle

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


def project(sp, ctx, K, Nc, Ns, *args, **kw):
    Kd = torch.from_numpy(np.array(K)).cuda()
    sp.sparkling_project(ctx, Kd, Nc, Ns, sp.make_proj(*args, **kw))
    sp.sparkling_status(ctx)
    return Kd.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("rows", [1, 2])
@pytest.mark.parametrize("c,d", [(0.25, 2.0 ** -26), (0.3, 2.0 ** -30), (0.25, 2.0 ** -34), (0.3, -2.0 ** -26)])
def test_a_row_at_its_radius(sp, ctx, c, d, rows, dt):
    """One row (a first or a second difference) of length c and a radius of
    c (1 - d): the first sample, 0 before, moves by c d / 2 or -c d / 6, which an
    FP32 result shows.  Gate: the two-float iteration's error, 2^-45 of the dual
    c / 20 an iteration, ten times in the fixed point's sum, below c 2^-44; a
    row that a comparison of the leading words took for inside leaves 0."""
    c = float(np.float32(c))
    Ns = rows + 1
    K = np.zeros((3 * Ns, 3), dt)
    K[rows::Ns, 1] = c
    r = [float("inf")] * 2
    r[rows - 1] = c * (1.0 - d)
    ref = oracle.project(K.astype(np.float64), 3, Ns, *r, n_iter=300)
    out = project(sp, ctx, K, 3, Ns, *r, 0.5, 300)
    assert d < 0 or abs(ref[0, 1]) > 0.1 * c * d      # away from or towards the last sample
    np.testing.assert_allclose(out[0::Ns], ref[0::Ns], rtol=2.0 ** -23, atol=c * 2.0 ** -44)


def walk(Ns, seed=0):
    return np.cumsum(np.random.default_rng(seed).normal(scale=0.02, size=(2, Ns, 3)), axis=1).reshape(-1, 3)


@pytest.mark.parametrize("Ns", [40, 600, 1100])
@pytest.mark.parametrize("e,tol", [(400, 1e-11), (-400, 1e-11), (-520, 1e-4)])
def test_fp64_samples_of_any_scale(sp, ctx, Ns, e, tol):
    """The projection of s K onto s times the set is s times the projection.  At
    2^-520 the squares are subnormal (2^-1054 and less: 20 bits and less of the
    smallest, 1e-4 of a dual)."""
    s = 2.0 ** e
    a, b = 1.0 / (2 * Ns), 1.0 / (8 * Ns * Ns)
    if e == -520:
        a, b = 0.01, 0.02                     # squares of 2^-1053 and up
    K = walk(Ns)
    ref = oracle.project(K, 2, Ns, a, b, n_iter=30)
    out = project(sp, ctx, K * s, 2, Ns, a * s, b * s, 0.5 * s, 30)
    np.testing.assert_allclose(out / s, ref, rtol=0, atol=tol)


def test_fp64_samples_whose_squares_overflow(sp, ctx):
    """1/|z| is 0 then: the row keeps its length, and stays finite."""
    out = project(sp, ctx, walk(40) * 2.0 ** 530, 2, 40, 2.0 ** 505, 2.0 ** 505, 2.0 ** 529, 30)
    assert np.isfinite(out).all() and np.abs(out).max() <= 2.0 ** 529


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("n_iter", [0, 1, 3, 40])
def test_not_a_number_spreads_as_the_rows_do(sp, ctx, dt, n_iter, sign):
    """Two samples an iteration to either side, in all components, of that shot."""
    K = walk(200).astype(dt)
    K[70, 1] = np.copysign(np.nan, sign)
    out = project(sp, ctx, K, 2, 200, 0.01, 1e-4, 0.5, n_iter)
    want = oracle.project(K.astype(np.float64), 2, 200, 0.01, 1e-4, n_iter=n_iter)
    np.testing.assert_array_equal(np.isnan(out), np.isnan(want))


@pytest.mark.parametrize("dt", [np.float32, np.float64])
def test_infinities_are_clipped(sp, ctx, dt):
    K = walk(200).astype(dt)
    K[70, 1], K[71, 2] = np.inf, -np.inf
    out = project(sp, ctx, K, 2, 200, 0.01, 1e-4, 0.5, 20)
    big = K.copy()
    big[70, 1], big[71, 2] = 1e18, -1e18      # beyond any dual's reach
    want = oracle.project(big.astype(np.float64), 2, 200, 0.01, 1e-4, n_iter=20)
    np.testing.assert_allclose(out, want, rtol=0, atol=1e-11 if dt == np.float64 else 2.0 ** -24)


@pytest.mark.parametrize("Nc,Ns,at", [(1, 300, 3), (2, 900, 899), (2, 1100, 5), (300, 40, 7), (40, 1300, 640), (400, 1300, 640)])
def test_not_a_number_reaches_the_other_ctas(sp, ctx, Nc, Ns, at):
    """One CTA, halos, clusters: the shot's other CTAs take part, other shots not."""
    K = np.cumsum(np.random.default_rng(Ns).normal(scale=0.002, size=(Nc, Ns, 3)), axis=1).reshape(-1, 3)
    K[at, 2] = np.nan
    a, b = 1.0 / (2 * Ns), 1.0 / (8 * Ns * Ns)
    out = project(sp, ctx, K, Nc, Ns, a, b, 0.5, 40)
    want = oracle.project(K, Nc, Ns, a, b, n_iter=40)
    np.testing.assert_array_equal(np.isnan(out), np.isnan(want))
    np.testing.assert_allclose(out, want, rtol=0, atol=1e-11)
