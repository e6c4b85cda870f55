"""Replayed evaluations of every kind (energy, forces, virial, dipoles alone,
several tolerances, more kinds than are kept), interleaved on one context with
new positions each time, before and after a change of the box or the batch:
each gives what a new context gives.  Bounds: FP64, with the solve at 1e-11 D,
1e-8 of the largest value (a warm start ends at other dipoles within the
tolerance); mixed, at 1e-7 D, the method's 1e-6 and 2e-5."""
import time

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


def _system(what):
    if what == "box":
        s, o = synth.make_config("water216")
        return s, dict(periodic=True, box=s.box, rc=o["rc"], grid=o["grid"], ewald_alpha=o["ewald"])
    if what == "batch":
        s, start, _ = synth.make_cluster_sizes([3, 40, 64, 12], seed=71)
        return s, dict(periodic=False, cluster_start=start)
    return synth.make_cluster(12, seed=51), dict(periodic=False)


@pytest.mark.parametrize("what", ["cluster", "batch", "box"])
@pytest.mark.parametrize("warm", [0, 1])
@pytest.mark.parametrize("prec", ["PREC_FP64", "PREC_MIXED"])
def test_every_kind(what, warm, prec, monkeypatch):
    import paper_2201_00804_gb300 as pkg
    monkeypatch.setenv("SIBFA_TUNE", "0")   # graphs are captured once the schedule is fixed
    s, kw = _system(what)
    fp64 = prec == "PREC_FP64"
    tol = 1e-11 if fp64 else 1e-7
    n = s.n_mol * 9

    def new(box=None, warm_start=0):
        return pkg.sibfa_create(synth.PARAMS, s.mp_local, pcg_tol_D=tol, precision=getattr(pkg, prec),
                                warm_start=warm_start, **(dict(kw, box=box) if box is not None else kw))

    def call(ctx, pos, kind, box=None):
        F, W = np.zeros(n), np.zeros((3, 3))
        b = {} if box is None else dict(box=np.array(box, dtype=np.float64))
        if kind == "energy":
            return [pkg.sibfa_energy_forces(ctx, pos, **b)["total"]]
        if kind == "forces":
            return [pkg.sibfa_energy_forces(ctx, pos, F, **b)["total"], F]
        if kind == "virial":
            return [pkg.sibfa_energy_forces(ctx, pos, F, virial=W, **b)["total"], F, W]
        pkg.sibfa_solve_dipoles(ctx, pos, F, kind * tol)
        return [F]

    rng = np.random.default_rng(52)
    ctx = new(warm_start=warm)

    def round_(kinds, box):
        for kind in kinds:
            move = np.repeat(rng.normal(0, 0.02, (s.n_mol, 1, 3)), 3, 1).reshape(-1)
            pos = np.ascontiguousarray(s.pos.reshape(-1) + move)
            got = call(ctx, pos, kind, None if isinstance(kind, (int, float)) else box)
            other = new(box)
            try:
                want = call(other, pos, kind)
            finally:
                pkg.sibfa_destroy(other)
            for k, (a, b) in enumerate(zip(got, want)):
                bound = 1e-8 if fp64 else (1e-6 if k == 0 and kind in ("energy", "forces", "virial") else 2e-5)
                if isinstance(kind, (int, float)):   # dipoles: 8 kind tol D either side, plus FP32's 1e-6 D
                    assert np.abs(a - b).max() * 4.80321 <= 16 * kind * tol * n ** 0.5 + (0 if fp64 else 2e-5), kind
                else:
                    assert np.abs(a - b).max() <= bound * max(1.0, np.abs(b).max()), (kind, k)

    try:
        full = ["forces", "virial", 1.0, "energy", 3.0]
        round_(full * 5, None)
        round_([1.0 + 0.25 * k for k in range(9)] * 3 + full * 4, None)   # more kinds than are kept
        if what == "box":
            for box in (s.box * 1.01, s.box):
                round_(full * 4, box)
    finally:
        pkg.sibfa_destroy(ctx)


def test_regrouped_batch(monkeypatch):
    """A job that stays in the server's batch while others come and go: the
    steps between are replayed, and each regrouping starts anew."""
    import torch
    import paper_2201_00804_gb300 as pkg
    monkeypatch.setenv("SIBFA_TUNE", "0")
    jobs = [(synth.make_cluster(4 + k, seed=400 + k), 150 if k == 0 else 6 + k) for k in range(8)]
    vel = [synth.maxwell_velocities(c, 300.0, seed=k) for k, (c, _) in enumerate(jobs)]
    srv = pkg.Server(synth.PARAMS, slots=1, batch_waters=256, precision=pkg.PREC_MIXED)
    try:
        tickets = []
        for (c, steps), v in zip(jobs, vel):
            tickets.append(srv.submit(c.pos, c.mp_local, periodic=False, n_steps=steps, vel=v, dt_fs=0.5))
            time.sleep(0.004)
        res, end = {}, time.time() + 120
        while len(res) < len(tickets):
            assert time.time() < end
            for t in tickets:
                if t not in res and (r := srv.poll(t)) is not None:
                    res[t] = r
    finally:
        srv.close()
    for (c, steps), v, t in zip(jobs, vel, tickets):
        ctx = pkg.sibfa_create(synth.PARAMS, c.mp_local, periodic=False, precision=pkg.PREC_MIXED, pcg_tol_D=1e-6,
                               warm_start=1)
        try:
            pos = torch.tensor(c.pos.reshape(-1), dtype=torch.float64, device="cuda")
            w = torch.tensor(v.reshape(-1), dtype=torch.float64, device="cuda")
            m = torch.tensor(c.masses().reshape(-1), dtype=torch.float64, device="cuda")
            e = pkg.sibfa_md_steps(ctx, pos, w, m, 0.5, steps)
        finally:
            pkg.sibfa_destroy(ctx)
        r = res[t]
        assert r["status"] == 0 and r["batched"]
        mag = sum(abs(e[k]) for k in ("elec", "pen", "rep", "disp", "xdisp", "pol", "ct"))
        assert abs(r["terms"]["total"] - e["total"]) <= 1e-6 * mag
        assert np.abs(r["pos"] - pos.cpu().numpy()).max() <= 1e-5
