"""One large cluster among thousands of single waters: how many molecules a
warp takes is laid out for the large cluster too, not for the mean size."""
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


def test_a_large_cluster_among_single_waters():
    """FP64.  The single waters have no pairs, so the batch's time is the large
    cluster's, give or take the launches (1.1 times; with warps filled by the mean size
    2.5 times, and 1.3 times that of the large cluster's earlier kernels).  Its
    terms and forces are those it has alone, to 1e-9 of their largest."""
    import torch
    import paper_2201_00804_gb300 as pkg
    big = synth.make_cluster(385, seed=91)
    one = synth.make_cluster(1, seed=92)
    out, best = [], []
    for extra in (0, 5000):
        pos = np.concatenate([big.pos.reshape(-1, 9)] + [one.pos.reshape(-1, 9)] * extra)
        mp = np.concatenate([big.mp_local] + [one.mp_local] * extra)
        pos = torch.tensor(pos.reshape(-1), dtype=torch.float64, device="cuda")
        F = torch.zeros_like(pos)
        kw = dict(cluster_start=np.concatenate([[0], 385 + np.arange(extra + 1)])) if extra else {}
        ctx = pkg.sibfa_create(synth.PARAMS, mp, periodic=False, precision=pkg.PREC_FP64, pcg_tol_D=1e-10,
                               warm_start=False, **kw)
        try:
            t = []
            for _ in range(20):
                t0 = time.perf_counter()
                pkg.sibfa_energy_forces(ctx, pos, F)
                t.append(time.perf_counter() - t0)
            terms = pkg.sibfa_cluster_terms(ctx, extra + 1)[0]
        finally:
            pkg.sibfa_destroy(ctx)
        best.append(min(t))
        out.append((terms, F.cpu().numpy()[:385 * 9]))
    (e0, F0), (e1, F1) = out
    mag = max(abs(v) for v in e0.values())
    assert all(abs(e0[k] - e1[k]) <= 1e-9 * mag for k in e0)
    assert np.abs(F0 - F1).max() <= 1e-9 * np.abs(F0).max()
    assert best[1] <= 1.7 * best[0], best
