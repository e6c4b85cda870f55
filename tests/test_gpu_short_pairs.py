"""Each molecule pair of the short-range terms, and each gas-phase pair of the
permanent energy, is evaluated by the molecule that the parity of their
indices names, in rounds that run across molecules."""
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


def _terms(sizes):
    import torch
    import paper_2201_00804_gb300 as pkg
    s, start, _ = synth.make_cluster_sizes(sizes, seed=21)
    ctx = pkg.sibfa_create(synth.PARAMS, s.mp_local, periodic=False, cluster_start=start, pcg_tol_D=1e-8,
                           precision=pkg.PREC_FP64, warm_start=False)
    try:
        pkg.sibfa_energy_forces(ctx, torch.tensor(s.pos.reshape(-1), dtype=torch.float64, device="cuda"))
        return pkg.sibfa_cluster_terms(ctx, len(sizes))
    finally:
        pkg.sibfa_destroy(ctx)


@pytest.mark.parametrize("sizes", [[2, 3, 31, 32, 33, 64, 65], [1, 200, 5], [385, 222]],
                         ids=["mixed", "large", "full"])
def test_rounds_across_molecules_agree(sizes):
    """The same clusters in batches of other sizes, whose warps take other
    numbers of molecules: the sums run in another order only, so each cluster's
    terms agree to 1e-12 of their magnitude (a few hundred FP64 additions of
    relative error 1e-16)."""
    a = _terms(sizes)
    b = _terms(sizes + [32] * 60)   # the same seeds for the first clusters
    for x, y in zip(a, b):
        mag = sum(abs(x[t]) for t in ("elec", "pen", "rep", "disp", "xdisp"))
        for t in ("elec", "pen", "rep", "disp", "xdisp"):
            assert abs(x[t] - y[t]) <= 1e-12 * mag, (t, x[t], y[t])


@pytest.mark.parametrize("prec,tol", [("PREC_FP64", 1e-9), ("PREC_MIXED", 2e-5)])
def test_order_of_molecules_does_not_matter(prec, tol):
    """658 waters at rc 11 in two orders.  In the second the last molecule has
    an odd index and its nearest 300 neighbours even ones, so all of its some 260
    pairs are another molecule's to evaluate: more rows than an inbox has.
    Energies and forces agree to the method's bounds of FP64 (1e-9 of the largest, with the
    solve at 1e-12) and FP32 (2e-5)."""
    import paper_2201_00804_gb300 as pkg
    s = synth.make_box(9, 27.2, seed=41, n_remove=71)
    assert s.n_mol == 658
    O = s.pos.reshape(-1, 3, 3)[:, 0]
    d = O - O[0]
    d -= s.box * np.round(d / s.box)
    near = np.argsort((d ** 2).sum(1))
    order = np.empty(658, dtype=int)
    order[657] = near[0]
    order[0:600:2] = near[1:301]
    order[np.r_[1:600:2, 600:657]] = near[301:]
    assert sorted(order) == list(range(658))
    out = []
    for perm in (np.arange(658), order):
        pos = np.ascontiguousarray(s.pos.reshape(658, 9)[perm])
        ctx = pkg.sibfa_create(synth.PARAMS, np.ascontiguousarray(s.mp_local[perm]), periodic=True, box=s.box, rc=11.0,
                               grid=32, ewald_alpha=0.35, pcg_tol_D=1e-12 if prec == "PREC_FP64" else 1e-7,
                               precision=getattr(pkg, prec), warm_start=False)
        F = np.zeros(658 * 9)
        try:
            e = pkg.sibfa_energy_forces(ctx, pos.reshape(-1), F)
        finally:
            pkg.sibfa_destroy(ctx)
        back = np.empty((658, 9))
        back[perm] = F.reshape(658, 9)
        out.append((e, back))
    (e0, f0), (e1, f1) = out
    mag = max(abs(e0[t]) for t in ("rep", "disp", "xdisp"))
    for t in ("rep", "disp", "xdisp"):
        assert abs(e0[t] - e1[t]) <= tol * mag, (t, e0[t], e1[t])
    assert np.abs(f0 - f1).max() <= tol * np.abs(f0).max()
