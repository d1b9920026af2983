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
