"""Boxes of few waters, whose one-kernel solve has blocks that own no molecule
and only transform, against the separate kernels (the host loop): dipoles to
8 times the tolerance (eigenvalues of 1 - alpha T of at least 0.25), in the mixed
path plus its dipole bound, forces to 1e-8 and 1e-5 of their norm."""
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


def _few(n, L, seed):
    """n waters of a lattice box of side L."""
    s = synth.make_box(6, L, seed=seed)
    keep = np.sort(np.random.default_rng(seed).permutation(s.n_mol)[:n])
    return synth.System(pos=np.ascontiguousarray(s.pos.reshape(-1, 9)[keep]).reshape(n, 3, 3),
                        mp_local=np.ascontiguousarray(s.mp_local[keep]), box=s.box)


@pytest.mark.parametrize("n,grid", [(1, (24, 24, 24)), (2, (25, 27, 30)), (9, (64, 24, 36)), (30, (64, 64, 64)),
                                    (30, (22, 24, 24)), (77, (96, 30, 32)), (153, (128, 24, 25))])
@pytest.mark.parametrize("fp64", [True, False])
def test_blocks_without_molecules(n, grid, fp64, monkeypatch):
    import paper_2201_00804_gb300 as pkg
    s = _few(n, 20.0, 30 + n)
    pos = np.ascontiguousarray(s.pos.reshape(-1))
    tol = 1e-9 if fp64 else 1e-7

    def run():
        ctx = pkg.sibfa_create(synth.PARAMS, s.mp_local, periodic=True, box=s.box, rc=7.0, grid=grid, ewald_alpha=0.4,
                               pcg_tol_D=tol, precision=pkg.PREC_FP64 if fp64 else pkg.PREC_MIXED, warm_start=False)
        mu, F = np.zeros_like(pos), np.zeros_like(pos)
        try:
            it, res = pkg.sibfa_solve_dipoles(ctx, pos, mu)
            pkg.sibfa_energy_forces(ctx, pos, F)
        finally:
            pkg.sibfa_destroy(ctx)
        return mu, F, it, res

    a = run()
    monkeypatch.setenv("SIBFA_PCG_HOST_LOOP", "1")
    b = run()
    rms = float(np.sqrt(((a[0] - b[0]) ** 2).sum() / (3 * n))) * 4.80321
    assert rms <= 8 * tol + (0.0 if fp64 else MIXED_MU_RMS_D), rms
    assert abs(a[2] - b[2]) <= 1 and a[3] < tol and b[3] < tol
    assert np.linalg.norm(a[1] - b[1]) <= (1e-8 if fp64 else 1e-5) * max(np.linalg.norm(b[1]), 1.0)
