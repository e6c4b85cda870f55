"""Device memory of a context: what nothing reads is not allocated, nor
charged when a server admits a job."""
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


def _bytes_of(create):
    import torch
    import paper_2201_00804_gb300 as pkg
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = create()
    try:
        return before - torch.cuda.mem_get_info()[0]
    finally:
        pkg.sibfa_destroy(ctx)


def test_clusters_that_solve_on_their_own_keep_no_pair_list(monkeypatch):
    """4096 clusters of 32 waters: the pair list has 20 bytes for each of a
    water's 3 x 3 x 31 atom pairs, 731 MB, and only the host-driven solve reads it."""
    import paper_2201_00804_gb300 as pkg
    M = 4096 * 32

    def create():
        return pkg.sibfa_create(synth.PARAMS, np.zeros((M, 5, 10)), periodic=False,
                                cluster_start=np.arange(0, M + 1, 32), precision=pkg.PREC_MIXED)

    pkg.sibfa_destroy(create())   # what a process allocates once
    own = _bytes_of(create)
    monkeypatch.setenv("SIBFA_PCG_HOST_LOOP", "1")
    listed = _bytes_of(create)
    assert listed - own > 0.95 * M * 9 * 31 * 20, (own, listed)


def test_admission_does_not_charge_a_list_that_is_not_kept():
    """A cluster of 64 waters is estimated at 96 MiB and 13,200 bytes a water;
    its pair list would be another 11,340 a water, above this cap."""
    import time
    import paper_2201_00804_gb300 as pkg
    s = synth.make_cluster(64, seed=64)
    srv = pkg.Server(synth.PARAMS, slots=1, batch_waters=0, precision=pkg.PREC_MIXED,
                     device_mem_bytes=(96 << 20) + 64 * (13200 + 11340 // 2))
    try:
        t = srv.submit(s.pos, s.mp_local, n_steps=0)
        end = time.time() + 60
        while (r := srv.poll(t)) is None:
            assert time.time() < end
            time.sleep(0.002)
        assert r["status"] == 0
    finally:
        srv.close()


@pytest.mark.parametrize("prec,tol", [("PREC_FP64", 1e-9), ("PREC_MIXED", 2e-5)])
def test_box_that_only_just_fits(prec, tol, monkeypatch):
    """A context that may not have all the memory it would take keeps fewer rows
    for the short-range gradients, down to none, and gives the same forces (to the
    bounds of FP64, with the solve at 1e-12, and of FP32, of the largest)."""
    import paper_2201_00804_gb300 as pkg
    s, o = synth.make_config("water216")
    pos = np.ascontiguousarray(s.pos.reshape(-1))
    kw = dict(periodic=True, box=s.box, rc=o["rc"], grid=o["grid"], ewald_alpha=o["ewald"],
              pcg_tol_D=1e-12 if prec == "PREC_FP64" else 1e-7, precision=getattr(pkg, prec), warm_start=False)

    def run():
        ctx = pkg.sibfa_create(synth.PARAMS, s.mp_local, **kw)
        F = np.zeros_like(pos)
        try:
            return pkg.sibfa_energy_forces(ctx, pos, F), F
        finally:
            pkg.sibfa_destroy(ctx)

    e0, F0 = run()
    rows = 216 * 70 * 16 * (8 if prec == "PREC_FP64" else 4)   # bytes of all rows at rc 7
    lo, hi = 1 << 20, 1 << 26   # the least bound under which creation succeeds
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        monkeypatch.setenv("SIBFA_MAX_DEVICE_BYTES", str(mid))
        try:
            pkg.sibfa_destroy(pkg.sibfa_create(synth.PARAMS, s.mp_local, **kw))
            hi = mid
        except pkg.SibfaError:
            lo = mid
    for bound in (hi, hi + rows // 4, hi + rows // 2, hi + rows):
        monkeypatch.setenv("SIBFA_MAX_DEVICE_BYTES", str(bound))
        e1, F1 = run()
        for t in ("rep", "disp", "xdisp"):
            assert abs(e0[t] - e1[t]) <= tol * abs(e0[t]), (bound, t)
        assert np.abs(F0 - F1).max() <= tol * np.abs(F0).max(), bound
