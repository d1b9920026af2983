"""What the calls ask of the context's workspace, read from the refusal under a
limit of one byte (nothing is launched)."""
import re

import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2108_02991_gb300 as sp
    return sp


def asked(sp, call):
    c = sp.sparkling_create(0)
    try:
        sp.sparkling_set_memory_limit(c, 1)
        with pytest.raises(sp.SparklingError) as e:
            call(c)
        assert e.value.code == sp.E_NOMEM
        return int(re.search(r"take the context to (\d+) bytes", str(e.value)).group(1))
    finally:
        c.close()


def samples(N, dt=torch.float32):
    return torch.zeros(N, 3, device="cuda", dtype=dt)


@pytest.mark.parametrize("tiles", [2, 20, 64])
def test_few_samples_ask_for_samples_and_totals(sp, tiles):
    """Within a number of tiles only the packed samples (16 bytes each) and the
    repulsion's totals (24) grow, up to the alignment of three arrays; not the
    block sums of the energy, 16 bytes for every 8 or 32 samples."""
    g = sp.make_grid(torch.from_numpy(inputs.density_gaussian(8, 0.2).rho).cuda())
    lo, hi = 1024 * (tiles - 1) + 1, 1024 * tiles
    for call in (lambda c, N: sp.sparkling_energy(c, samples(N), g),
                 lambda c, N: sp.sparkling_grad(c, samples(N), g)):
        more = asked(sp, lambda c: call(c, hi)) - asked(sp, lambda c: call(c, lo))
        assert more <= (hi - lo) * 40 + 3 * 256


def test_projections_in_a_second_launch_ask_for_no_state(sp):
    """FP32 trajectories of 2560 samples a shot: as items (FP64 asked for) every
    CTA of the engine has a state of 18 doubles a sample, in the second launch
    none has."""
    rho = torch.from_numpy(inputs.density_gaussian(8, 0.2).rho).cuda()
    K = samples(4 * 2560)
    pr = sp.make_proj(1e-3, 1e-5, 0.5, 5)

    def call(c, mode):
        sp.sparkling_set_projection(c, mode)
        sp.sparkling_step_batched(c, K, [0, 4 * 2560], 2560, [sp.make_grid(rho)], [1e-5], [pr])

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    items = asked(sp, lambda c: call(c, sp.PROJECTION_FP64))
    assert items - asked(sp, lambda c: call(c, sp.PROJECTION_DEFAULT)) >= sms * 18 * 8 * 2560
