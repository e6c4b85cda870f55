"""The polarization solve in one kernel against the separate kernels (the host
loop) on the same inputs: system sizes around the blocks' shares, grids of
every radix, wrapped and unaligned rows, a grid with another prime (which
takes the separate kernels), and the gas phase.  Both solve T mu = E to the
same residual; with eigenvalues of alpha T of at least 0.25 in these systems
two solutions differ by at most 8 tol RMS, plus in the mixed path the FP32
rounding of the products, held to the mixed path's dipole bound."""
import numpy as np
import pytest

import synth
from gpu_util import MIXED_MU_RMS_D

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_00804_gb300 import build
    build.build()


def _mu(pkg, s, kw, tol, prec):
    import torch
    ctx = pkg.sibfa_create(synth.PARAMS, s.mp_local, pcg_tol_D=tol, precision=prec, warm_start=False, **kw)
    try:
        pos = torch.tensor(s.pos.reshape(-1), dtype=torch.float64, device="cuda")
        mu = torch.zeros_like(pos)
        it, res = pkg.sibfa_solve_dipoles(ctx, pos, mu)
        F = torch.zeros_like(pos)
        e = pkg.sibfa_energy_forces(ctx, pos, F)
        torch.cuda.synchronize()
        return mu.cpu().numpy(), it, res, e, F.cpu().numpy()
    finally:
        pkg.sibfa_destroy(ctx)


CASES = [("box", (6, 6, 6), (24, 24, 24)), ("box", (6, 7, 6), (25, 27, 30)), ("box", (7, 6, 6), (32, 45, 36)),
         ("box", (6, 6, 8), (22, 24, 32)), ("box", (8, 9, 9), (30, 54, 50)), ("box", (12, 11, 12), (48, 64, 60)),
         ("gas", 1, None), ("gas", 2, None), ("gas", 33, None), ("gas", 200, None)]


@pytest.mark.parametrize("kind,size,grid", CASES)
@pytest.mark.parametrize("fp64", [True, False])
def test_one_kernel_matches_the_separate_kernels(kind, size, grid, fp64, monkeypatch):
    import paper_2201_00804_gb300 as pkg
    if kind == "box":
        s = synth.make_ortho_box(size, tuple(3.11 * n for n in size), seed=11)
        kw = dict(periodic=True, box=s.box, rc=7.0, grid=grid, ewald_alpha=0.4)
    else:
        s = synth.make_cluster(size, seed=12)
        kw = dict(periodic=False)
    tol = 1e-9 if fp64 else 1e-7
    prec = pkg.PREC_FP64 if fp64 else pkg.PREC_MIXED
    a = _mu(pkg, s, kw, tol, prec)
    monkeypatch.setenv("SIBFA_PCG_HOST_LOOP", "1")
    b = _mu(pkg, s, kw, tol, prec)
    rms = float(np.sqrt(((a[0] - b[0]) ** 2).sum() / (a[0].size / 3))) * 4.80321
    assert rms <= 8 * tol + (0.0 if fp64 else MIXED_MU_RMS_D), rms
    assert abs(a[1] - b[1]) <= 1 and a[2] < tol and b[2] < tol
    f = np.linalg.norm(a[4] - b[4]) / max(np.linalg.norm(b[4]), 1e-30)
    assert f <= (1e-8 if fp64 else 1e-5), f


@pytest.mark.parametrize("sizes", [[1], [1, 2, 3, 42, 43, 64], [2] * 40 + [5, 8, 11, 21, 22, 32], [64, 64, 1]])
def test_clusters_on_their_own_match_the_batch_solve(sizes, monkeypatch):
    """Mixed path: each cluster's own solve (lanes per row from 16 down to 1,
    clusters up to the largest it takes) against the batch-wide one."""
    import paper_2201_00804_gb300 as pkg
    s, start, _ = synth.make_cluster_sizes(sizes, seed=31)
    kw = dict(periodic=False) if len(sizes) == 1 else dict(periodic=False, cluster_start=start)
    tol = 1e-7
    a = _mu(pkg, s, kw, tol, pkg.PREC_MIXED)
    monkeypatch.setenv("SIBFA_PCG_HOST_LOOP", "1")
    b = _mu(pkg, s, kw, tol, pkg.PREC_MIXED)
    for c in range(len(sizes)):
        x, y = (v[0][start[c] * 9:start[c + 1] * 9] for v in (a, b))
        assert float(np.sqrt(((x - y) ** 2).sum() / (x.size / 3))) * 4.80321 <= 8 * tol + MIXED_MU_RMS_D, c
    assert a[2] < tol
    assert np.linalg.norm(a[4] - b[4]) <= 1e-5 * max(np.linalg.norm(b[4]), 1e-30)


def test_iteration_limit_is_reported():
    import paper_2201_00804_gb300 as pkg
    s, o = synth.make_config("water216")
    kw = dict(periodic=True, box=s.box, rc=o["rc"], grid=o["grid"], ewald_alpha=0.4, pcg_max_iter=3)
    with pytest.raises(pkg.SibfaError) as err:
        _mu(pkg, s, kw, 1e-9, pkg.PREC_FP64)
    assert err.value.status == -3
