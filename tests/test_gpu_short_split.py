"""FP64 short-range kernels with a molecule's list shared by four warps (small
systems) against one warp a molecule (larger ones): the same clusters in a
batch below and above the line between the two.  The sums run in another
order only, so each cluster's repulsion and dispersion agree to 1e-12 of
their magnitude (a few hundred FP64 additions of relative error 1e-16)."""
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


@pytest.mark.parametrize("sizes", [[2, 3, 31, 32, 33, 64, 65], [1, 200, 5], [607]], ids=["mixed", "large", "full"])
def test_shared_and_whole_lists_agree(sizes):
    if len(sizes) == 1:
        sizes = [385, 222]   # 607 waters: the largest shared system
    pad = [32] * ((608 - sum(sizes) + 31) // 32)
    a = _terms(sizes)
    b = _terms(sizes + pad)   # the same seeds for the first clusters
    for x, y in zip(a, b):
        mag = sum(abs(x[t]) for t in ("rep", "disp", "xdisp"))
        for t in ("rep", "disp", "xdisp"):
            assert abs(x[t] - y[t]) <= 1e-12 * mag, (t, x[t], y[t])
