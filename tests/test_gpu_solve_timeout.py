"""A wait between the blocks of the one-kernel solve that runs out: the call
says so, and the next one works and starts from the direct field (same results
and as many iterations as a new context)."""
import numpy as np
import pytest

import synth
from gpu_util import TERMS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_00804_gb300 import build
    build.build()


@pytest.mark.parametrize("prec", ["PREC_FP64", "PREC_MIXED"])
@pytest.mark.parametrize("warm", [0, 1, 4])
@pytest.mark.parametrize("periodic", [True, False], ids=["box", "gas"])
def test_a_wait_that_runs_out(periodic, warm, prec, monkeypatch):
    import paper_2201_00804_gb300 as pkg
    monkeypatch.setenv("SIBFA_TUNE", "0")   # replayed graphs from the third call on
    if periodic:
        s, o = synth.make_config("water216")
        kw = dict(periodic=True, box=s.box, rc=o["rc"], grid=o["grid"], ewald_alpha=o["ewald"])
    else:
        s, kw = synth.make_cluster(100, seed=61), dict(periodic=False)
    fp64 = prec == "PREC_FP64"
    tol = 1e-10 if fp64 else 1e-7
    pos = np.ascontiguousarray(s.pos.reshape(-1))

    def new():
        return pkg.sibfa_create(synth.PARAMS, s.mp_local, pcg_tol_D=tol, precision=getattr(pkg, prec), warm_start=warm,
                                **kw)

    def call(ctx):
        F = np.zeros_like(pos)
        e = pkg.sibfa_energy_forces(ctx, pos, F)
        return e, F, pkg.sibfa_last_stats(ctx)[0]

    other = new()
    try:
        e0, F0, it0 = call(other)
    finally:
        pkg.sibfa_destroy(other)
    ctx = new()
    try:
        for _ in range(5):
            call(ctx)
        for k in range(2):
            pkg.sibfa_set_wait_polls(ctx, 0)
            for what in (lambda: call(ctx), lambda: pkg.sibfa_solve_dipoles(ctx, pos, np.zeros_like(pos), tol)):
                with pytest.raises(pkg.SibfaError) as err:
                    what()
                assert err.value.status == -6
            pkg.sibfa_set_wait_polls(ctx, 1 << 22)
            e, F, it = call(ctx)
            assert it == it0
            mag = sum(abs(e0[t]) for t in TERMS)
            assert all(abs(e[t] - e0[t]) <= (1e-11 if fp64 else 1e-6) * mag for t in TERMS)
            assert np.abs(F - F0).max() <= (1e-9 if fp64 else 2e-5) * np.abs(F0).max()
    finally:
        pkg.sibfa_destroy(ctx)
