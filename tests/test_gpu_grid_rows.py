"""Grids whose z rows are a multiple of four points, even and odd: the FP32
spread adds a stencil row as four-wide, two-wide or single reductions, wrapped
rows one by one.  Against the FP64 path, which adds every point singly, to the
FP32 bound of 2e-5 of the largest force."""
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


@pytest.mark.parametrize("grid", [24, 26, 27])
def test_mixed_forces_match_fp64(grid):
    import paper_2201_00804_gb300 as pkg
    s, o = synth.make_config("water216")
    F = []
    for prec, tol in ((pkg.PREC_FP64, 1e-10), (pkg.PREC_MIXED, 1e-7)):
        ctx = pkg.sibfa_create(synth.PARAMS, s.mp_local, periodic=True, box=s.box, rc=o["rc"], grid=grid,
                               ewald_alpha=o["ewald"], pcg_tol_D=tol, precision=prec, warm_start=False)
        f = np.zeros(s.n_mol * 9)
        try:
            pkg.sibfa_energy_forces(ctx, np.ascontiguousarray(s.pos.reshape(-1)), f)
        finally:
            pkg.sibfa_destroy(ctx)
        F.append(f)
    assert np.abs(F[0] - F[1]).max() <= 2e-5 * np.abs(F[0]).max()
