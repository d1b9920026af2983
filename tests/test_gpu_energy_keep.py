"""The differentiable energy's forward and backward, call by call: what the
forward launches and holds, and whose settings the backward takes.

Gates: value and gradient against the separate calls as in
test_gpu_energy_and_grad.py (the same FP32 terms, grouped differently: 2e-6);
where the backward sums the attraction itself it is the separate call, bit for
bit.
"""
import re

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


@pytest.fixture
def ctx(sp):
    c = sp.sparkling_create(0)
    yield c
    c.close()


def problem(sp, N, dt=torch.float32):
    rng = np.random.default_rng(N)
    K = torch.from_numpy((0.3 * rng.normal(size=(N, 3))).clip(-0.5, 0.5)).cuda().to(dt)
    rho = torch.from_numpy(inputs.density_gaussian(12, 0.2, 0.1).rho).cuda()
    return K, rho, sp.make_grid(rho)


def launches(sp, ctx, fn):
    """Launch scopes by kind of one call, after a first one that tunes."""
    fn()
    sp.sparkling_set_timing(ctx, True)
    sp.sparkling_kernel_times(ctx, reset=True)
    fn()
    torch.cuda.synchronize()
    t = sp.sparkling_kernel_times(ctx, reset=True)
    sp.sparkling_set_timing(ctx, False)
    return t["attraction"][1], t["repulsion"][1]


@pytest.mark.parametrize("acc", [0, 1])
@pytest.mark.parametrize("N", [2, 1000, 25000])
def test_each_sum_once(sp, ctx, N, acc):
    """The forward sums the repulsion once (its energy), the backward once (its
    force) and the attraction not again; without keeping, as the separate calls."""
    K, rho, g = problem(sp, N)
    K.requires_grad_(True)
    assert launches(sp, ctx, lambda: sp.sparkling_energy_fn(K, rho, ctx, acc=acc)) == (1, 1)
    F = sp.sparkling_energy_fn(K, rho, ctx, acc=acc)
    assert launches(sp, ctx, lambda: torch.autograd.grad(F, K, retain_graph=True)) == (0, 1)
    F2 = sp.sparkling_energy_fn(K, rho, ctx, acc=acc, keep_attraction=False)
    assert launches(sp, ctx, lambda: torch.autograd.grad(F2, K, retain_graph=True)) == (1, 1)
    E = sp.sparkling_energy(ctx, K.detach(), g, acc)[0]
    d = sp.sparkling_energy_backward(ctx, K.detach(), g, acc=acc)
    assert float(F2.detach()) == E and float(F.detach()) == pytest.approx(E, rel=2e-6)
    (a,), (b,) = torch.autograd.grad(F, K), torch.autograd.grad(F2, K)
    assert torch.equal(b, d)
    assert rel_l2(a.cpu().numpy(), d.cpu().numpy()) < 2e-6


@pytest.mark.parametrize("N", [1000, 25000])
def test_no_more_workspace_than_the_separate_calls(sp, N):
    K, rho, g = problem(sp, N, torch.float64)
    K.requires_grad_(True)
    c = sp.sparkling_create(0)
    sp.sparkling_set_memory_limit(c, 1)
    with pytest.raises(sp.SparklingError) as e:
        sp.sparkling_energy(c, K.detach(), g)
    need = int(re.search(r"take the context to (\d+) bytes", str(e.value)).group(1))
    try:
        sp.sparkling_set_memory_limit(c, need)
        (a,) = torch.autograd.grad(sp.sparkling_energy_fn(K, rho, c), K)
        sp.sparkling_status(c)
        sp.sparkling_set_memory_limit(c, 0)
        assert rel_l2(a.cpu().numpy(), sp.sparkling_energy_backward(c, K.detach(), g).cpu().numpy()) < 2e-6
    finally:
        c.close()


def test_the_backward_takes_the_settings_of_its_call(sp, ctx):
    K, rho, g = problem(sp, 3000)
    K.requires_grad_(True)
    F = sp.sparkling_energy_fn(K, rho, ctx)
    for change in (lambda: sp.sparkling_set_regularisation(ctx, 0.05),
                   lambda: sp.sparkling_set_attraction(ctx, sp.ATTRACTION_FIELD)):
        change()
        (a,) = torch.autograd.grad(F, K, retain_graph=True)
        assert torch.equal(a, sp.sparkling_energy_backward(ctx, K.detach(), g))
    sp.sparkling_set_attraction(ctx, sp.ATTRACTION_DIRECT)
    sp.sparkling_set_regularisation(ctx, 0.0)
    assert launches(sp, ctx, lambda: torch.autograd.grad(F, K, retain_graph=True)) == (0, 1)


def test_modes_that_keep_nothing(sp, ctx):
    K, rho, g = problem(sp, 3000)
    assert sp.sparkling_keeps_attraction(ctx, sp.ACC_KAHAN32)
    assert not sp.sparkling_keeps_attraction(ctx, sp.ACC_FP64_PAIR)
    E, A, eps = sp.sparkling_energy_keep(ctx, K, g, sp.ACC_FP64_PAIR)
    assert A is None and eps == -1.0 and E == sp.sparkling_energy(ctx, K, g, sp.ACC_FP64_PAIR)
    K.requires_grad_(True)
    (a,) = torch.autograd.grad(sp.sparkling_energy_fn(K, rho, ctx, acc=sp.ACC_FP64_PAIR), K)
    assert torch.equal(a, sp.sparkling_energy_backward(ctx, K.detach(), g, acc=sp.ACC_FP64_PAIR))
    A = torch.empty(3000, 3, device="cuda")
    with pytest.raises(TypeError):
        sp.sparkling_energy_backward_kept(ctx, K.detach(), g, A, 0.0)
    with pytest.raises(ValueError):
        sp.sparkling_energy_backward_kept(ctx, K.detach(), g, A[:5].double(), 0.0)


def attraction_ms(sp, ctx, fn, reps=6):
    fn()
    sp.sparkling_set_timing(ctx, True)
    sp.sparkling_kernel_times(ctx, reset=True)
    for _ in range(reps):
        fn()
    torch.cuda.synchronize()
    t = sp.sparkling_kernel_times(ctx, reset=True)["attraction"]
    sp.sparkling_set_timing(ctx, False)
    return t[0] / t[1]


@pytest.mark.parametrize("shape", [0, 1, 2])
def test_the_combined_pass_is_near_the_force_in_every_shape(sp, ctx, shape):
    """Both bound by one reciprocal square root a pair: the combined kernel has
    one multiply-add more and fewer resident CTAs.  1.35 times the force's time
    is the gate (a third of the CTAs gone at worst); registers capped for CTAs
    that shared memory does not hold made it 1.85 at 128 threads."""
    K = torch.rand(65536, 3, device="cuda", generator=torch.Generator("cuda").manual_seed(3)) - 0.5
    rho = torch.from_numpy(inputs.density_gaussian(48, 0.2, 0.1).rho).cuda()
    g = sp.make_grid(rho)
    sp.sparkling_set_shape(ctx, "attraction", shape)
    G = torch.empty_like(K)
    force = attraction_ms(sp, ctx, lambda: sp.sparkling_grad(ctx, K, g, 0, G))
    both = attraction_ms(sp, ctx, lambda: sp.sparkling_energy_keep(ctx, K, g))
    assert both < 1.35 * force
