"""Mixed path: every cluster's dipoles leave a residual below the tolerance,
also where waters pressed together give alpha T eigenvalues below -1 (at which a
Jacobi step leads away from the solution)."""
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


def _alpha_T(x):
    """alpha times the Thole-damped dipole field matrix between the atoms of different waters, x (n, 3, 3)."""
    P, n = synth.PARAMS, len(x)
    a = np.tile([P["alpha_o"], P["alpha_h"], P["alpha_h"]], n)
    mol = np.repeat(np.arange(n), 3)
    d = x.reshape(-1, 3)[:, None] - x.reshape(-1, 3)[None]
    r = np.sqrt((d ** 2).sum(-1) + np.eye(3 * n))
    u = P["thole"] * r ** 3 / np.sqrt(a[:, None] * a[None])
    t1, t2 = (1 - np.exp(-u)) / r ** 3, 3 * (1 - (1 + u) * np.exp(-u)) / r ** 5
    T = t2[..., None, None] * d[..., :, None] * d[..., None, :] - t1[..., None, None] * np.eye(3)
    T[mol[:, None] == mol[None]] = 0
    return np.repeat(a, 3)[:, None] * T.transpose(0, 2, 1, 3).reshape(9 * n, 9 * n)


@pytest.mark.parametrize("squeeze", [1.0, 0.6, 0.4])
def test_residual_of_every_cluster(squeeze):
    """alpha times the residual of the returned dipoles, (1 - alpha T)(mu - mu*),
    with mu* the mixed path's own solution at 1e-9 D (where atoms nearly touch, at
    0.4, the FP32 kernels shift the solution itself by up to 6e-5 D, whichever solve
    is taken).  The rounding of the vectors adds some 1e-7 of fields up to 100 D."""
    import paper_2201_00804_gb300 as pkg
    sizes = [4, 8, 16, 32, 64] * 16
    s, start, _ = synth.make_cluster_sizes(sizes, seed=73)
    x = s.pos.reshape(-1, 3, 3)
    x = x + (squeeze - 1.0) * x[:, :1]   # O nearer to the origin, waters as they are
    pos = np.ascontiguousarray(x.reshape(-1))

    def dipoles(tol):
        ctx = pkg.sibfa_create(synth.PARAMS, s.mp_local, periodic=False, cluster_start=start,
                               precision=pkg.PREC_MIXED, warm_start=False, pcg_max_iter=400)
        mu = np.zeros_like(pos)
        try:
            pkg.sibfa_solve_dipoles(ctx, pos, mu, tol)
        finally:
            pkg.sibfa_destroy(ctx)
        return mu

    solved = dipoles(1e-9)
    M = [_alpha_T(x[start[c]:start[c + 1]]) for c in range(len(sizes))]
    for tol in (1e-2, 1e-3):
        e = dipoles(tol) - solved
        worst = 0.0
        for c, n in enumerate(sizes):
            v = e[start[c] * 9:start[c + 1] * 9]
            z = v - M[c] @ v
            worst = max(worst, np.sqrt((z ** 2).sum() / (3 * n)) * 4.80321)
        assert worst <= tol * 1.001 + 1e-5, (tol, worst)
