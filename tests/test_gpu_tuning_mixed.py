"""The mixed path has one schedule of its short-range kernel (its registers cap
the blocks per SM already, and finishing it before the solve only loses), so
there is nothing to time and no cap to report, from the first call on."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_00804_gb300 import build
    build.build()


@pytest.mark.parametrize("periodic", [True, False], ids=["box", "gas"])
def test_one_schedule_and_no_cap(periodic):
    import paper_2201_00804_gb300 as pkg
    if periodic:
        s, o = synth.make_config("water216")
        kw = dict(periodic=True, box=s.box, rc=o["rc"], grid=o["grid"], ewald_alpha=o["ewald"])
    else:
        s, kw = synth.make_cluster(12, seed=51), dict(periodic=False)
    pos = np.ascontiguousarray(s.pos.reshape(-1))
    ctx = pkg.sibfa_create(synth.PARAMS, s.mp_local, precision=pkg.PREC_MIXED, warm_start=False, **kw)
    try:
        for _ in range(16):
            assert pkg.sibfa_tuned_shape(ctx) == (0, True)
            assert pkg.sibfa_tuned_schedule(ctx) == (0, False, True, [0.0] * 5)
            pkg.sibfa_energy_forces(ctx, pos)
    finally:
        pkg.sibfa_destroy(ctx)
