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


def shots(Nc, Ns, seed, spread=0.02, through=None):
    """Random walks; through=(m, p): sample m of every shot near p (a pin that is
    far away leaves hundreds of iterations unsettled, and a rounding error of the
    input grows a thousandfold and more)."""
    rng = np.random.default_rng(seed)
    K = np.cumsum(rng.normal(scale=spread, size=(Nc, Ns, 3)), axis=1)
    if through is None:
        K += rng.uniform(-0.4, 0.4, size=(Nc, 1, 3))
    else:
        m, p = through
        K += np.asarray(p) + rng.normal(scale=1e-3, size=(Nc, 1, 3)) - K[:, m:m + 1]
    return np.clip(K, -0.5, 0.5).reshape(-1, 3).astype(np.float32)


PIN = (0.1, 0.2, -0.3)


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


def batch(sp, Ns, counts, alpha, beta, n_iter, dt=np.float32):
    Ks, grids, projs, etas, refs = [], [], [], [], []
    for b, c in enumerate(counts):
        g = inputs.density_gaussian(8 + 3 * b, 0.2, 0.1)
        K = shots(c, Ns, 100 * Ns + b, 0.2 / Ns, (Ns - 1, PIN) if b == 1 else None).astype(dt)
        a, be = (alpha, beta) if alpha else ((0.5 + b) / (2 * Ns), (0.5 + b) / (8 * Ns * Ns))
        pin, eta = (Ns - 1 if b == 1 else -1), 0.3 / (c * Ns)
        Ks.append(K)
        grids.append(sp.make_grid(torch.from_numpy(g.rho).cuda(), g.lo, g.hi, g.n))
        projs.append(sp.make_proj(a, be, 0.5, n_iter, pin, PIN))
        etas.append(eta)
        refs.append(oracle.step(K.astype(np.float64), c, Ns, g, eta, a, be, 0.5, pin, PIN, n_iter))
    return Ks, np.concatenate([[0], np.cumsum([k.shape[0] for k in Ks])]), grids, projs, etas, refs


def check_batch(sp, ctx, Ns, counts, alpha, beta, n_iter, one_launch, graph, mixed):
    Ks, off, grids, projs, etas, refs = batch(sp, Ns, counts, alpha, beta, n_iter)
    for _ in range(3 if graph else 1):        # eager, captured, replayed
        K = torch.from_numpy(np.concatenate(Ks)).cuda()
        sp.sparkling_step_batched(ctx, K, off, Ns, grids, etas, projs, one_launch=one_launch, graph=graph)
        sp.sparkling_status(ctx)
        out = K.cpu().numpy()
        for b in range(len(Ks)):
            tol = (proj_tol_f32(refs[b], Ks[b]) if mixed else PROJ_F32_ROUND) + 4 * etas[b] * GRAD_ABS
            np.testing.assert_allclose(out[off[b]:off[b + 1]], refs[b].astype(np.float32), rtol=0, atol=tol)


# what keeps FP32 trajectories out of the two-float form: more iterations than
# its table, radii below its range, FP64 asked for
FALLBACKS = [("iterations", None, None, 4097), ("radii", 1e-14, 1e-16, 30), ("asked", None, None, 30)]


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("one_launch", [False, True])
@pytest.mark.parametrize("mode,what,alpha,beta,n_iter", [("fp64", *f) for f in FALLBACKS] +
                         [("mixed", *FALLBACKS[1])])       # its bound is one of tens of iterations
def test_fp32_projection_items_of_the_engine(sp, ctx, mode, what, alpha, beta, n_iter, one_launch, graph):
    """Shots whose state fits shared memory; pins on the last sample."""
    if what == "asked":
        sp.sparkling_set_projection(ctx, sp.PROJECTION_FP64)
    elif mode == "mixed":
        sp.sparkling_set_projection(ctx, sp.PROJECTION_MIXED)
    check_batch(sp, ctx, 96, [3, 11, 1], alpha, beta, n_iter, one_launch, graph, mode == "mixed")


@pytest.mark.parametrize("one_launch", [False, True])
@pytest.mark.parametrize("mode", ["fp64", "mixed"])
def test_fp32_projection_items_with_state_in_global_memory(sp, ctx, mode, one_launch):
    """Longer than the register form takes, and than shared memory holds."""
    if mode == "mixed":
        sp.sparkling_set_projection(ctx, sp.PROJECTION_MIXED)
    check_batch(sp, ctx, 8193, [1, 2], None, None, 20, one_launch, False, mode == "mixed")


def test_a_change_of_form_rebuilds_the_plan(sp, ctx):
    """The same batch, graph-replayed, in the second launch, as items, and back."""
    for n_iter in (30, 30, 30, 4097, 4097, 30, 30):
        check_batch(sp, ctx, 64, [2, 5], None, None, n_iter, True, True, False)
    sp.sparkling_set_projection(ctx, sp.PROJECTION_FP64)
    check_batch(sp, ctx, 64, [2, 5], None, None, 30, True, True, False)
    sp.sparkling_set_projection(ctx, sp.PROJECTION_DEFAULT)
    check_batch(sp, ctx, 64, [2, 5], None, None, 30, True, True, False)


@pytest.mark.parametrize("Nc,Ns,pin", [(40, 33, 0), (9, 512, 256), (3, 700, 699)])
def test_mixed_form_with_state_in_shared_memory(sp, ctx, Nc, Ns, pin):
    """The FP32 iteration on the displacement, where the slew radius is below the
    two-float form's range."""
    K = shots(Nc, Ns, Ns, 0.2 / Ns, (pin, PIN))
    a, b = 1.0 / (2 * Ns), 1e-14
    ref = oracle.project(K.astype(np.float64), Nc, Ns, a, b, pin_index=pin, pin=PIN, n_iter=60)
    sp.sparkling_set_projection(ctx, sp.PROJECTION_MIXED)
    Kd = torch.from_numpy(K).cuda()
    sp.sparkling_project(ctx, Kd, Nc, Ns, sp.make_proj(a, b, 0.5, 60, pin, PIN))
    out = Kd.cpu().numpy()
    np.testing.assert_allclose(out, ref.astype(np.float32), rtol=0, atol=proj_tol_f32(ref, K))
    np.testing.assert_array_equal(out.reshape(Nc, Ns, 3)[:, pin],
                                  np.broadcast_to(np.float32(PIN), (Nc, 3)))


@pytest.mark.parametrize("Nc,Ns,pin", [(9, 512, 256), (3, 2560, 1280)])
def test_mixed_is_two_float_in_its_range(sp, ctx, Nc, Ns, pin):
    K = shots(Nc, Ns, Ns, 2e-3)
    a, b = 1.0 / (2 * Ns), 1.0 / (8 * Ns * Ns)
    ref = oracle.project(K.astype(np.float64), Nc, Ns, a, b, pin_index=pin, n_iter=60)
    sp.sparkling_set_projection(ctx, sp.PROJECTION_MIXED)
    Kd = torch.from_numpy(K).cuda()
    sp.sparkling_project(ctx, Kd, Nc, Ns, sp.make_proj(a, b, 0.5, 60, pin))
    np.testing.assert_allclose(Kd.cpu().numpy(), ref.astype(np.float32), rtol=0, atol=PROJ_F32_ROUND)


@pytest.mark.parametrize("form", ["second launch", "items"])
@pytest.mark.parametrize("one_launch", [False, True])
def test_fp32_timeout_leaves_trajectories_alone(sp, ctx, form, one_launch):
    """With a zero wait budget projection items cannot wait for pair items, and
    the step reports it (the second launch waits for nothing: there only a copy
    could run out, and need not).  Every shot is projected in full or left
    alone, and with the default budget the same context gives the result bit for
    bit."""
    if form == "items":
        sp.sparkling_set_projection(ctx, sp.PROJECTION_FP64)
    Ks, off, grids, projs, etas, refs = batch(sp, 256, [24, 9, 31], None, None, 30)
    K0 = np.concatenate(Ks)

    def run():
        K = torch.from_numpy(K0).cuda()
        sp.sparkling_step_batched(ctx, K, off, 256, grids, etas, projs, one_launch=one_launch, graph=False)
        return K

    ref = run()
    sp.sparkling_status(ctx)
    ref = ref.cpu().numpy()
    for b in range(3):
        np.testing.assert_allclose(ref[off[b]:off[b + 1]], refs[b].astype(np.float32), rtol=0,
                                   atol=PROJ_F32_ROUND + 4 * etas[b] * GRAD_ABS)
    sp.sparkling_set_wait_budget(ctx, 0)
    out = run()
    code = sp.OK
    try:
        sp.sparkling_status(ctx)
    except sp.SparklingError as e:
        code = e.code
    assert code == sp.E_TIMEOUT or (form == "second launch" and code == sp.OK)
    out = out.cpu().numpy()
    assert code == sp.E_TIMEOUT or (out == ref).all()
    for b in range(3):
        s = slice(off[b], off[b + 1])
        # shot by shot: left alone, or the full result
        got, was, want = (x[s].reshape(-1, 768) for x in (out, K0, ref))
        same = (got == was).all(axis=1)
        assert (same | (got == want).all(axis=1)).all()
    sp.sparkling_set_wait_budget(ctx, -1)
    again = run()
    sp.sparkling_status(ctx)
    np.testing.assert_array_equal(again.cpu().numpy(), ref)
