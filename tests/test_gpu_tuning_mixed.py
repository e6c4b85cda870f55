"""The schedule tuning of the mixed path.  Its short-range kernel takes no cap
on the blocks per SM, so there are two schedules to try, and no cap to report."""
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
def test_two_schedules_and_no_cap(periodic, monkeypatch):
    import paper_2201_00804_gb300 as pkg
    if periodic:
        s, o = synth.make_config("water216")
        kw = dict(periodic=True, box=s.box, rc=o["rc"], grid=o["grid"], ewald_alpha=o["ewald"])
    else:
        s, kw = synth.make_cluster(12, seed=51), dict(periodic=False)
    pos = np.ascontiguousarray(s.pos.reshape(-1))
    ctx = pkg.sibfa_create(synth.PARAMS, s.mp_local, precision=pkg.PREC_MIXED, warm_start=False, **kw)
    try:
        assert pkg.sibfa_tuned_shape(ctx) == (0, False)
        for _ in range(11):   # 2 warm-up + 2 schedules x 4 timed, each read at the next call
            pkg.sibfa_energy_forces(ctx, pos)
        blocks, join, done, ms = pkg.sibfa_tuned_schedule(ctx)
        assert done and blocks == 0 and pkg.sibfa_tuned_shape(ctx) == (0, True)
        assert [t > 0 for t in ms] == [False, True, False, True, False]
        assert join == (ms[3] < ms[1])
    finally:
        pkg.sibfa_destroy(ctx)
    monkeypatch.setenv("SIBFA_TUNE", "0")
    ctx = pkg.sibfa_create(synth.PARAMS, s.mp_local, precision=pkg.PREC_MIXED, warm_start=False, **kw)
    try:
        assert pkg.sibfa_tuned_schedule(ctx)[:3] == (0, False, True)
    finally:
        pkg.sibfa_destroy(ctx)
