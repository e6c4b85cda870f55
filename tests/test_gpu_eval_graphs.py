"""Evaluations of small systems replay captured graphs from the third call of
a kind on: every call has to give what a new context gives.  FP64, with the
solve at 1e-11, so both agree to 1e-9 of the largest force and of the energy."""
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


@pytest.mark.parametrize("periodic", [False, True], ids=["cluster", "box"])
def test_replayed_calls_match_a_new_context(periodic, monkeypatch):
    import paper_2201_00804_gb300 as pkg
    monkeypatch.setenv("SIBFA_TUNE", "0")   # graphs are captured once the schedule is fixed
    if periodic:
        s, o = synth.make_config("water216")
        kw = dict(periodic=True, box=s.box, rc=o["rc"], grid=o["grid"], ewald_alpha=o["ewald"])
    else:
        s, kw = synth.make_cluster(12, seed=51), dict(periodic=False)

    def new():
        return pkg.sibfa_create(synth.PARAMS, s.mp_local, pcg_tol_D=1e-11, precision=pkg.PREC_FP64, warm_start=False,
                                **kw)

    def run(ctx, pos, kind):
        F = np.zeros(s.n_mol * 9)
        if kind == "energy":
            return pkg.sibfa_energy_forces(ctx, pos)["total"], F
        return pkg.sibfa_energy_forces(ctx, pos, F)["total"], F

    rng = np.random.default_rng(52)
    ctx = new()
    try:
        for call in range(12):
            pos = np.ascontiguousarray(s.pos.reshape(-1) + np.repeat(rng.normal(0, 0.02, (s.n_mol, 1, 3)), 3, 1).reshape(-1))
            kind = "energy" if call % 3 == 2 else "forces"
            e, F = run(ctx, pos, kind)
            other = new()
            try:
                e0, F0 = run(other, pos, kind)
            finally:
                pkg.sibfa_destroy(other)
            assert abs(e - e0) <= 1e-9 * abs(e0), call
            assert np.abs(F - F0).max() <= 1e-9 * max(np.abs(F0).max(), 1.0), call
    finally:
        pkg.sibfa_destroy(ctx)
